// CUDA-core implicit-GEMM convolution (forward, input gradient, weight
// gradient) with fp32 accumulation.  This is the fp32 compute path of the
// library (the fp32 tiny workload) and serves layers whose shapes the
// tensor-core kernels do not take (e.g. a first layer of 3 channels).
//
// All three passes are one tiled GEMM C[M][N] = sum_k A[M][k] B[k][N] whose
// operands are gathered on the fly from NHWC tensors:
//   FWD    M = output pixels, N = Co, k = (r, s, ci):  A = x window, B = w
//   DGRAD  M = input pixels,  N = Ci, k = (r, s, co):  A = dy (strided), B = w
//   WGRAD  M = Co, N = (r, s, ci), k = output pixel:   A = dy^T, B = x window
//
// What bounds it: these are small problems on a fraction of the chip, so the
// time is the serial chain of k-tiles of one block.  Hence two shared-memory
// buffers with the next tile's loads in flight during the products (one
// barrier per k-tile of 32, 16 for the widest tile), four operand values per load and one window
// decomposition per load (32-bit, hoisted for the index that is fixed per
// thread), micro-tiles read as 16-byte vectors, and tiles narrow enough to
// spread small outputs over the SMs.  Per launch in a profiled step (event
// pair included), against one 64 x 64 tile kernel with 64-bit index arithmetic
// per element: fp32 16 x 16 x 16, 32 -> 64 channels, forward 62.7 -> 18.2 us
// and weight gradient 42.8 -> 18.3; bf16 64 x 32 x 32, 3 -> 128 channels,
// forward 53 -> 29 and weight gradient 125 -> 37.
#pragma once
#include "fo_common.cuh"
#include "fo_kernels.h"

#include <algorithm>

namespace fo {
namespace simt {

enum Mode { FWD = 0, DGRAD = 1, WGRAD = 2 };

constexpr int NT = 256;

struct Geo {
  int N, H, W, Ci, Co, k, stride, pad, Ho, Wo;
  int M, Ncol, K;
  int ntiles; // column tiles; blockIdx.x runs over (row tile, column tile), columns fastest
  int kper;   // k-range per blockIdx.z (K split); the output of split z starts at c + z * M * Ncol
};

// Four consecutive elements (the address is a multiple of four elements).
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const bf16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const bf16* e = reinterpret_cast<const bf16*>(&u);
  return make_float4(__bfloat162float(e[0]), __bfloat162float(e[1]), __bfloat162float(e[2]), __bfloat162float(e[3]));
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(bf16* p, const float (&v)[4]) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&lo);
  u.y = *reinterpret_cast<uint32_t*>(&hi);
  *reinterpret_cast<uint2*>(p) = u;
}
__device__ __forceinline__ float& at(float4& v, int i) { return reinterpret_cast<float*>(&v)[i]; }

// A pixel index split into image, row and column of an Hh x Ww grid.
struct Pix {
  int n, h, w;
};
__device__ __forceinline__ Pix pixel(int p, int Hh, int Ww) {
  const unsigned t = unsigned(p) / unsigned(Ww);
  return {int(t / unsigned(Hh)), int(t % unsigned(Hh)), int(unsigned(p) % unsigned(Ww))};
}
// Tap index rs of a k x k window (k is 1 or 3): row and column.
__device__ __forceinline__ int tap_row(int rs, int k) { return k == 1 ? 0 : (rs * 11) >> 5; }

// The operand's element at (index fixed per thread, k): see load_a / load_b.
// x[n][h][w][ci] of output pixel q under tap (r, s), or null outside.
template <typename T>
__device__ __forceinline__ const T* x_at(const Geo& g, const T* x, const Pix& q, int rs, int ci) {
  const int r = tap_row(rs, g.k), s = rs - r * g.k;
  const int h = q.h * g.stride + r - g.pad, w = q.w * g.stride + s - g.pad;
  if (unsigned(h) >= unsigned(g.H) || unsigned(w) >= unsigned(g.W)) return nullptr;
  return x + ((int64_t(q.n) * g.H + h) * g.W + w) * g.Ci + ci;
}
// dy[n][ho][wo][co] that tap (r, s) carries into input pixel q, or null.
template <typename T>
__device__ __forceinline__ const T* dy_at(const Geo& g, const T* dy, const Pix& q, int rs, int co) {
  const int r = tap_row(rs, g.k), s = rs - r * g.k;
  int h = q.h + g.pad - r, w = q.w + g.pad - s;
  if (h < 0 || w < 0) return nullptr;
  if (g.stride == 2) {
    if ((h | w) & 1) return nullptr;
    h >>= 1;
    w >>= 1;
  }
  if (h >= g.Ho || w >= g.Wo) return nullptr;
  return dy + ((int64_t(q.n) * g.Ho + h) * g.Wo + w) * g.Co + co;
}

// Four operand values.  FWD / DGRAD, A: row m (pixel q), k .. k + 3; FWD, B:
// column n, k .. k + 3; DGRAD, B and WGRAD: four consecutive columns (rows)
// from m at one k.  V: the four are contiguous in memory and all valid or all
// out of range (the channel count they run over is a multiple of 4).
template <int MODE, bool V, typename TA>
__device__ __forceinline__ float4 load_a(const Geo& g, const TA* a, int m, const Pix& q, int k, int kend) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (MODE == WGRAD) {   // A[co][p] = dy[p][co]
    if (k >= kend) return v;
    const TA* p = a + int64_t(k) * g.Co + m;
    if (V) {
      if (m < g.M) v = ld4(p);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (m + i < g.M) at(v, i) = to_f(p[i]);
    }
    return v;
  }
  if (m >= g.M) return v;
  const int ch = MODE == FWD ? g.Ci : g.Co;
  if (V) {
    if (k >= kend) return v;
    const int rs = unsigned(k) / unsigned(ch), c = k - rs * ch;
    const TA* p = MODE == FWD ? x_at(g, a, q, rs, c) : dy_at(g, a, q, rs, c);
    if (p) v = ld4(p);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (k + i >= kend) break;
      const int rs = unsigned(k + i) / unsigned(ch), c = k + i - rs * ch;
      const TA* p = MODE == FWD ? x_at(g, a, q, rs, c) : dy_at(g, a, q, rs, c);
      if (p) at(v, i) = to_f(*p);
    }
  }
  return v;
}
template <int MODE, bool V, typename TB>
__device__ __forceinline__ float4 load_b(const Geo& g, const TB* b, int n, int k, int kend) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (MODE == FWD) {   // w[co][(r, s, ci)], four k
    if (n >= g.Ncol) return v;
    const TB* p = b + int64_t(n) * g.K + k;
    if (V) {
      if (k < kend) v = ld4(p);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k + i < kend) at(v, i) = to_f(p[i]);
    }
    return v;
  }
  if (k >= kend) return v;
  if (MODE == DGRAD) {   // w[co][r][s][ci], four ci
    const int rs = unsigned(k) / unsigned(g.Co), co = k - rs * g.Co;
    const TB* p = b + (int64_t(co) * g.k * g.k + rs) * g.Ci + n;
    if (V) {
      if (n < g.Ncol) v = ld4(p);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (n + i < g.Ncol) at(v, i) = to_f(p[i]);
    }
    return v;
  }
  const Pix q = pixel(k, g.Ho, g.Wo);   // WGRAD: x window of output pixel k, four (r, s, ci)
  if (V) {
    if (n < g.Ncol) {
      const int rs = unsigned(n) / unsigned(g.Ci);
      const TB* p = x_at(g, b, q, rs, n - rs * g.Ci);
      if (p) v = ld4(p);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (n + i >= g.Ncol) break;
      const int rs = unsigned(n + i) / unsigned(g.Ci);
      const TB* p = x_at(g, b, q, rs, n + i - rs * g.Ci);
      if (p) at(v, i) = to_f(*p);
    }
  }
  return v;
}

// BM x BN output tile, TM x TN outputs per thread (16-byte vectors of TN);
// the grid is (row tiles, column tiles, K splits).
template <int MODE, int BM, int BN, int BK, int TM, int TN, bool VA, bool VB, typename TA, typename TB, typename TC>
__global__ void __launch_bounds__(NT) simt_conv_kernel(Geo g, const TA* __restrict__ a, const TB* __restrict__ b,
                                                       const float* __restrict__ bias, TC* __restrict__ c, int relu,
                                                       int acc, const TC* __restrict__ mask) {
  static_assert((BM / TM) * (BN / TN) == NT, "thread tile");
  constexpr int PA = BM + 4, PB = BN + 4;          // shared-memory pitches (16-byte aligned rows)
  constexpr int QA = BM * BK / 4 / NT, QB = (BN * BK / 4 + NT - 1) / NT;   // loads per thread and k-tile
  static_assert(QA >= 1 && QB >= 1, "tile");
  constexpr int KQ = BK / 4;
  constexpr bool AK = MODE != WGRAD;               // A loads run along k (else along m)
  constexpr bool BKK = MODE == FWD;                // B loads run along k (else along n)
  __shared__ __align__(16) float As[2][BK][PA];
  __shared__ __align__(16) float Bs[2][BK][PB];
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x;
  const int m0 = int(blockIdx.x / unsigned(g.ntiles)) * BM, n0 = int(blockIdx.x % unsigned(g.ntiles)) * BN;
  const int kb = blockIdx.z * g.kper, ke = min(g.K, kb + g.kper);
  c += int64_t(blockIdx.z) * g.M * g.Ncol;

  Pix q[QA];
  if (AK)
#pragma unroll
    for (int i = 0; i < QA; ++i)
      q[i] = MODE == FWD ? pixel(m0 + (tid + i * NT) / KQ, g.Ho, g.Wo) : pixel(m0 + (tid + i * NT) / KQ, g.H, g.W);

  float4 ra[QA], rb[QB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < QA; ++i) {
      const int e = tid + i * NT;
      ra[i] = AK ? load_a<MODE, VA>(g, a, m0 + e / KQ, q[i], k0 + 4 * (e % KQ), ke)
                 : load_a<MODE, VA>(g, a, m0 + 4 * (e % (BM / 4)), q[0], k0 + e / (BM / 4), ke);
    }
#pragma unroll
    for (int i = 0; i < QB; ++i) {
      const int e = tid + i * NT;
      if (BN * BK / 4 % NT == 0 || e < BN * BK / 4)
        rb[i] = BKK ? load_b<MODE, VB>(g, b, n0 + e / KQ, k0 + 4 * (e % KQ), ke)
                    : load_b<MODE, VB>(g, b, n0 + 4 * (e % (BN / 4)), k0 + e / (BN / 4), ke);
    }
  };
  auto put = [&](int s) {
#pragma unroll
    for (int i = 0; i < QA; ++i) {
      const int e = tid + i * NT;
      if (AK)
#pragma unroll
        for (int j = 0; j < 4; ++j) As[s][4 * (e % KQ) + j][e / KQ] = at(ra[i], j);
      else
        *reinterpret_cast<float4*>(&As[s][e / (BM / 4)][4 * (e % (BM / 4))]) = ra[i];
    }
#pragma unroll
    for (int i = 0; i < QB; ++i) {
      const int e = tid + i * NT;
      if (BN * BK / 4 % NT != 0 && e >= BN * BK / 4) continue;
      if (BKK)
#pragma unroll
        for (int j = 0; j < 4; ++j) Bs[s][4 * (e % KQ) + j][e / KQ] = at(rb[i], j);
      else
        *reinterpret_cast<float4*>(&Bs[s][e / (BN / 4)][4 * (e % (BN / 4))]) = rb[i];
    }
  };

  const int tx = tid % (BN / TN), ty = tid / (BN / TN);
  float sum[TM][TN] = {};
  fetch(kb);
  put(0);
  __syncthreads();
  int s = 0;
  for (int k0 = kb; k0 < ke; k0 += BK, s ^= 1) {
    const bool more = k0 + BK < ke;
    if (more) fetch(k0 + BK);
#pragma unroll 8
    for (int kk = 0; kk < BK; ++kk) {
      float av[TM], bv[TN];
      if constexpr (TM % 4 == 0) {
#pragma unroll
        for (int i = 0; i < TM; i += 4) *reinterpret_cast<float4*>(&av[i]) = *reinterpret_cast<const float4*>(&As[s][kk][ty * TM + i]);
      } else {
#pragma unroll
        for (int i = 0; i < TM; i += 2) *reinterpret_cast<float2*>(&av[i]) = *reinterpret_cast<const float2*>(&As[s][kk][ty * TM + i]);
      }
      // columns tx * 4 + {0..3} of each BN / (TN / 4) wide part
#pragma unroll
      for (int j = 0; j < TN; j += 4)
        *reinterpret_cast<float4*>(&bv[j]) = *reinterpret_cast<const float4*>(&Bs[s][kk][j * (BN / TN) + tx * 4]);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) sum[i][j] = fmaf(av[i], bv[j], sum[i][j]);
    }
    if (more) {
      put(s ^ 1);   // its readers passed the barrier of the previous k-tile
      __syncthreads();
    }
  }
  const bool vec = g.Ncol % 4 == 0;   // whole four-wide accesses
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i;
    if (m >= g.M) continue;
#pragma unroll
    for (int jj = 0; jj < TN; jj += 4) {
      const int n = n0 + jj * (BN / TN) + tx * 4;
      const int64_t idx = int64_t(m) * g.Ncol + n;
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] = sum[i][jj + j];
        if (bias && n + j < g.Ncol) v[j] += bias[n + j];
        if (relu) v[j] = fmaxf(v[j], 0.f);
      }
      if (vec) {
        if (n >= g.Ncol) continue;
        if (mask) {
          float4 mk = ld4(mask + idx);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (!(at(mk, j) > 0.f)) v[j] = 0.f;
        }
        if (acc) {
          float4 o = ld4(c + idx);
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] += at(o, j);
        }
        st4(c + idx, v);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (n + j >= g.Ncol) continue;
          if (mask && !(to_f(mask[idx + j]) > 0.f)) v[j] = 0.f;
          if (acc) v[j] += to_f(c[idx + j]);
          c[idx + j] = from_f<TC>(v[j]);
        }
      }
    }
  }
}

// Tiles: 128 x 128 (8 x 8 outputs per thread, the most products per shared
// load) and 64 x 64 where at least one block per SM remains, 128 x 32 for
// narrow outputs (a first layer's weight gradient: 27 columns), else 32 x 64.
struct TileShape {
  int bm, bn;
};
TileShape tile_of(const Geo& g, int mode);

template <int MODE, bool VA, bool VB, typename TA, typename TB, typename TC>
void launch(Geo g, const void* a, const void* b, const float* bias, void* c, bool relu, bool acc, cudaStream_t st,
            const void* mask) {
  const TileShape t = tile_of(g, MODE);
  g.ntiles = ceil_div(g.Ncol, t.bn);
  const dim3 grid(unsigned(ceil_div(g.M, t.bm)) * unsigned(g.ntiles), 1, unsigned(ceil_div(g.K, g.kper)));
  auto go = [&](auto kernel) {
    launch_k(kernel, grid, NT, 0, st, g, (const TA*)a, (const TB*)b, bias, (TC*)c, relu ? 1 : 0, acc ? 1 : 0,
             (const TC*)mask);
  };
  if (t.bn == 32) go(simt_conv_kernel<MODE, 128, 32, 32, 4, 4, VA, VB, TA, TB, TC>);
  else if (t.bm == 128) go(simt_conv_kernel<MODE, 128, 128, 16, 8, 8, VA, VB, TA, TB, TC>);
  else if (t.bm == 64) go(simt_conv_kernel<MODE, 64, 64, 32, 4, 4, VA, VB, TA, TB, TC>);
  else if constexpr (MODE != WGRAD) go(simt_conv_kernel<MODE, 32, 64, 32, 2, 4, VA, VB, TA, TB, TC>);
}

// The operand types the server uses (the uploaded or stored activations, their
// gradients, and either weight copy), with four-wide loads where the channels
// they run over allow it.
template <int MODE, typename TA, typename TB, typename TC>
void launch_v(const Geo& g, const void* a, const void* b, const float* bias, void* c, bool relu, bool acc,
              cudaStream_t st, const void* mask) {
  const bool ci4 = g.Ci % 4 == 0, co4 = g.Co % 4 == 0;
  const bool va = MODE == FWD ? ci4 : co4, vb = ci4;
  if (va && vb) launch<MODE, true, true, TA, TB, TC>(g, a, b, bias, c, relu, acc, st, mask);
  else if (va && MODE != FWD) launch<MODE, MODE != FWD, false, TA, TB, TC>(g, a, b, bias, c, relu, acc, st, mask);
  else launch<MODE, false, false, TA, TB, TC>(g, a, b, bias, c, relu, acc, st, mask);
}
template <int MODE>
void launch_any(const Geo& g, const void* a, int dta, const void* b, int dtb, const float* bias, void* c, int dtc,
                bool relu, bool acc, cudaStream_t st, const void* mask = nullptr) {
  if (dta == kF32 && dtb == kF32 && dtc == kF32)
    return launch_v<MODE, float, float, float>(g, a, b, bias, c, relu, acc, st, mask);
  if constexpr (MODE == FWD) {   // hidden layers; the fp32 logits of the bf16 path
    if (dtc == kBF16) launch_v<MODE, bf16, bf16, bf16>(g, a, b, bias, c, relu, acc, st, mask);
    else launch_v<MODE, bf16, float, float>(g, a, b, bias, c, relu, acc, st, mask);
  } else if constexpr (MODE == DGRAD) {
    if (dta == kBF16) launch_v<MODE, bf16, bf16, bf16>(g, a, b, bias, c, relu, acc, st, mask);
    else launch_v<MODE, float, float, bf16>(g, a, b, bias, c, relu, acc, st, mask);
  } else {
    if (dta == kBF16) launch_v<MODE, bf16, bf16, float>(g, a, b, bias, c, relu, acc, st, mask);
    else launch_v<MODE, float, bf16, float>(g, a, b, bias, c, relu, acc, st, mask);
  }
}

// One translation unit per mode (k_simt_conv_fwd.cu and so on): they compile side by side.
void launch_fwd(const Geo& g, const void* a, int dta, const void* b, int dtb, const float* bias, void* c, int dtc,
                bool relu, cudaStream_t st);
void launch_dgrad(const Geo& g, const void* a, int dta, const void* b, int dtb, void* c, int dtc, bool acc,
                  cudaStream_t st, const void* mask);
void launch_wgrad(const Geo& g, const void* a, int dta, const void* b, int dtb, void* c, cudaStream_t st);

}  // namespace simt
}  // namespace fo
