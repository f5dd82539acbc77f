// Kernels of the MobileNetV3 bottleneck (the MobileNetV3-Large server part
// of Table 4): depthwise convolution, hard swish, hard sigmoid and the
// squeeze-and-excite channel scaling.  Activations are NHWC in fp32 or bf16
// (template parameter T); every arithmetic step runs in fp32.  Channels are
// the fastest index of every thread mapping, so a warp's loads and stores are
// contiguous.  Parameter gradients are written as per-chunk partials that a
// later batched launch sums in chunk order (no atomics: deterministic).
#include "fo_common.cuh"
#include "fo_kernels.h"

#include <algorithm>

namespace fo {

namespace {

#define FO_MB_DISPATCH(dt, T, ...) \
  do {                             \
    if ((dt) == kF32) {            \
      using T = float;             \
      __VA_ARGS__;                 \
    } else {                       \
      using T = bf16;              \
      __VA_ARGS__;                 \
    }                              \
  } while (0)

#define FO_MB_GRID_STRIDE(i, n) \
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < (n); i += int64_t(gridDim.x) * blockDim.x)

template <typename T>
__device__ __forceinline__ void store_acc(T* p, int64_t i, float v, bool acc) {
  if (acc) v += to_f(p[i]);
  p[i] = from_f<T>(v);
}

// --------------------------------------------------------- depthwise conv
// KT is the kernel size when known at compile time (3 or 5: the tap loops
// unroll, so a thread's loads are independent), or 0 for a runtime d.k.

// y[n,i,j,c] = b[c] + sum_{r,s} xpad[n, i*st + r, j*st + s, c] * w[c,r,s],
// w [C][k][k] in the activation type (the bf16 path multiplies the bf16
// copy of the weights), zero padding `pad` on each side.
template <typename T, int KT>
__global__ void __launch_bounds__(256) dwconv_fwd_k(const T* __restrict__ x, const T* __restrict__ w,
                                                    const float* __restrict__ bias, T* __restrict__ y,
                                                    DwShape d) {
  pdl_wait();
  pdl_trigger();
  const int K = KT ? KT : d.k;
  const int64_t n_out = int64_t(d.N) * d.Ho * d.Wo * d.C;
  FO_MB_GRID_STRIDE(idx, n_out) {
    const int c = int(idx % d.C);
    const int64_t p = idx / d.C;
    const int j = int(p % d.Wo);
    const int i = int((p / d.Wo) % d.Ho);
    const int64_t n = p / (int64_t(d.Wo) * d.Ho);
    const T* wc = w + int64_t(c) * K * K;
    float acc = bias ? bias[c] : 0.f;
#pragma unroll
    for (int r = 0; r < (KT ? KT : K); ++r) {
      const int h = i * d.stride - d.pad + r;
      if (h < 0 || h >= d.H) continue;
#pragma unroll
      for (int s = 0; s < (KT ? KT : K); ++s) {
        const int ww = j * d.stride - d.pad + s;
        if (ww < 0 || ww >= d.W) continue;
        acc = fmaf(to_f(x[((n * d.H + h) * d.W + ww) * d.C + c]), to_f(wc[r * K + s]), acc);
      }
    }
    y[idx] = from_f<T>(acc);
  }
}

// dx[n,h,w,c] (+)= sum over the taps (r,s) whose output position
// i = (h + pad - r) / st, j = (w + pad - s) / st is whole and in range of
// dy[n,i,j,c] * w[c,r,s].
template <typename T, int KT>
__global__ void __launch_bounds__(256) dwconv_dgrad_k(const T* __restrict__ dy, const T* __restrict__ w,
                                                      T* __restrict__ dx, DwShape d, int acc_flag) {
  pdl_wait();
  pdl_trigger();
  const int K = KT ? KT : d.k;
  const int64_t n_in = int64_t(d.N) * d.H * d.W * d.C;
  FO_MB_GRID_STRIDE(idx, n_in) {
    const int c = int(idx % d.C);
    const int64_t p = idx / d.C;
    const int wx = int(p % d.W);
    const int h = int((p / d.W) % d.H);
    const int64_t n = p / (int64_t(d.W) * d.H);
    const T* wc = w + int64_t(c) * K * K;
    float acc = 0.f;
#pragma unroll
    for (int r = 0; r < (KT ? KT : K); ++r) {
      const int ti = h + d.pad - r;
      if (ti < 0 || ti % d.stride) continue;
      const int i = ti / d.stride;
      if (i >= d.Ho) continue;
#pragma unroll
      for (int s = 0; s < (KT ? KT : K); ++s) {
        const int tj = wx + d.pad - s;
        if (tj < 0 || tj % d.stride) continue;
        const int j = tj / d.stride;
        if (j >= d.Wo) continue;
        acc = fmaf(to_f(dy[((n * d.Ho + i) * d.Wo + j) * d.C + c]), to_f(wc[r * K + s]), acc);
      }
    }
    store_acc(dx, idx, acc, acc_flag != 0);
  }
}

// Weight (and bias) gradient partials: chunk q of the output pixels
// [q * per, min(rows, (q + 1) * per)) gives
//   pw[q][c*k*k + r*k + s] = sum_p dy[p,c] * xpad[p's window at (r,s), c]
//   pb[q][c]               = sum_p dy[p,c]            (when pb is given)
// A block covers 32 channels (lane = channel) of one chunk; its 8 warps take
// every 8th pixel of the chunk with the k*k tap sums in registers, and the
// warps' sums are added in warp order through shared memory.
template <typename T, int KT>
__global__ void __launch_bounds__(256) dwconv_wgrad_k(const T* __restrict__ dy, const T* __restrict__ x,
                                                      float* __restrict__ pw, float* __restrict__ pb, DwShape d,
                                                      int per) {
  pdl_wait();
  pdl_trigger();
  constexpr int KK = KT * KT;
  __shared__ float red[8][KK + 1][33];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int c = blockIdx.x * 32 + lane;
  const int64_t rows = int64_t(d.N) * d.Ho * d.Wo;
  const int64_t p0 = int64_t(blockIdx.y) * per;
  const int64_t p1 = p0 + per < rows ? p0 + per : rows;
  float acc[KK + 1];
#pragma unroll
  for (int t = 0; t <= KK; ++t) acc[t] = 0.f;
  if (c < d.C) {
    for (int64_t p = p0 + warp; p < p1; p += 8) {
      const int j = int(p % d.Wo);
      const int i = int((p / d.Wo) % d.Ho);
      const int64_t n = p / (int64_t(d.Wo) * d.Ho);
      const float g = to_f(dy[p * d.C + c]);
      acc[KK] += g;
#pragma unroll
      for (int r = 0; r < KT; ++r) {
        const int h = i * d.stride - d.pad + r;
        if (h < 0 || h >= d.H) continue;
#pragma unroll
        for (int s = 0; s < KT; ++s) {
          const int ww = j * d.stride - d.pad + s;
          if (ww < 0 || ww >= d.W) continue;
          acc[r * KT + s] = fmaf(g, to_f(x[((n * d.H + h) * d.W + ww) * d.C + c]), acc[r * KT + s]);
        }
      }
    }
  }
#pragma unroll
  for (int t = 0; t <= KK; ++t) red[warp][t][lane] = acc[t];
  __syncthreads();
  const int c0 = blockIdx.x * 32;
  for (int e = threadIdx.x; e < 32 * (KK + 1); e += 256) {
    // e = (channel, tap): consecutive threads write consecutive floats of pw
    const int cl = e / (KK + 1), t = e % (KK + 1);
    if (c0 + cl >= d.C) continue;
    float sum = 0.f;
#pragma unroll
    for (int w8 = 0; w8 < 8; ++w8) sum += red[w8][t][cl];
    if (t < KK) pw[int64_t(blockIdx.y) * d.C * KK + int64_t(c0 + cl) * KK + t] = sum;
    else if (pb) pb[int64_t(blockIdx.y) * d.C + c0 + cl] = sum;
  }
}

// Any kernel size: one thread per (tap, channel) and chunk.
template <typename T>
__global__ void __launch_bounds__(256) dwconv_wgrad_any_k(const T* __restrict__ dy, const T* __restrict__ x,
                                                          float* __restrict__ pw, float* __restrict__ pb, DwShape d,
                                                          int per) {
  pdl_wait();
  pdl_trigger();
  const int kk = d.k * d.k;
  const int taps = kk + (pb ? 1 : 0);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= taps * d.C) return;
  const int c = t % d.C, tap = t / d.C;
  const int64_t rows = int64_t(d.N) * d.Ho * d.Wo;
  const int64_t p0 = int64_t(blockIdx.y) * per;
  const int64_t p1 = p0 + per < rows ? p0 + per : rows;
  float acc = 0.f;
  if (tap < kk) {
    const int r = tap / d.k, s = tap % d.k;
    for (int64_t p = p0; p < p1; ++p) {
      const int j = int(p % d.Wo);
      const int i = int((p / d.Wo) % d.Ho);
      const int64_t n = p / (int64_t(d.Wo) * d.Ho);
      const int h = i * d.stride - d.pad + r, ww = j * d.stride - d.pad + s;
      if (h < 0 || h >= d.H || ww < 0 || ww >= d.W) continue;
      acc = fmaf(to_f(dy[p * d.C + c]), to_f(x[((n * d.H + h) * d.W + ww) * d.C + c]), acc);
    }
    pw[int64_t(blockIdx.y) * d.C * kk + int64_t(c) * kk + tap] = acc;
  } else {
    for (int64_t p = p0; p < p1; ++p) acc += to_f(dy[p * d.C + c]);
    pb[int64_t(blockIdx.y) * d.C + c] = acc;
  }
}

// ------------------------------------------- depthwise conv, 8 channels wide
// The bf16 kernels for k = 3, 5 and channel counts that are multiples of 8:
// a thread owns 8 channels (one 16-byte access per tap), a block 64 channels,
// whose weights it stages once as fp32 [tap][channel].  The scalar kernels
// above read a channel's k * k weights with a stride of k * k elements and
// divide 64-bit indices per element, which bounded them.  Steps, us, with the
// scalar kernels and with these: MobileNet part on 4 x 4 maps at batch 64 372
// and 350, on 14 x 14 maps at batch 32 1065 and 745.
constexpr int kDwC = 64;        // channels per block
constexpr int kDwV = kDwC / 8;  // threads over them

struct F8 {
  float v[8];
};
__device__ __forceinline__ F8 up8(const uint4& u) {
  const bf16* e = reinterpret_cast<const bf16*>(&u);
  F8 r;
#pragma unroll
  for (int j = 0; j < 8; ++j) r.v[j] = __bfloat162float(e[j]);
  return r;
}
__device__ __forceinline__ F8 ld8(const bf16* p) { return up8(*reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ void st8(bf16* p, const F8& r) {
  uint4 u;
  bf16* e = reinterpret_cast<bf16*>(&u);
#pragma unroll
  for (int j = 0; j < 8; ++j) e[j] = __float2bfloat16_rn(r.v[j]);
  *reinterpret_cast<uint4*>(p) = u;
}
// a += x * w where `in`; else a as it is, also where w or x is not finite (a
// zero in their place would give NaN).
__device__ __forceinline__ void fma8(F8& a, const F8& x, const F8& w, bool in) {
#pragma unroll
  for (int j = 0; j < 8; ++j) a.v[j] = in ? fmaf(x.v[j], w.v[j], a.v[j]) : a.v[j];
}
__device__ __forceinline__ F8 ld8(const float* p) {
  const float4 u = *reinterpret_cast<const float4*>(p), v = *reinterpret_cast<const float4*>(p + 4);
  return {{u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w}};
}

// Block (channel block, pixel block of 16): DGRAD false, y = conv(x) + bias;
// DGRAD true, y = dx (+)= conv^T(x = dy).  A tap outside the map loads the
// first pixel and drops it, so that no branch keeps the loads of the taps
// from being in flight together.
constexpr int kDwThreads = 16 * kDwV;
template <int KT, bool DGRAD>
__global__ void __launch_bounds__(kDwThreads) dwconv_x8_k(const bf16* __restrict__ x, const bf16* __restrict__ w,
                                                          const float* __restrict__ bias, bf16* __restrict__ y,
                                                          DwShape d, unsigned rows, int acc_flag) {
  pdl_wait();
  pdl_trigger();
  constexpr int KK = KT * KT;
  __shared__ __align__(16) float ws[KK][kDwC + 4];
  const int c0 = blockIdx.x * kDwC, nc = min(kDwC, d.C - c0);
#pragma unroll 4
  for (int e = threadIdx.x; e < nc * KK; e += kDwThreads)
    ws[e % KK][e / KK] = __bfloat162float(w[int64_t(c0) * KK + e]);
  __syncthreads();
  const int cv = 8 * (threadIdx.x % kDwV), c = c0 + cv;
  if (cv >= nc) return;
  const unsigned Hy = DGRAD ? d.H : d.Ho, Wy = DGRAD ? d.W : d.Wo;   // the grid of y
  const int Hx = DGRAD ? d.Ho : d.H, Wx = DGRAD ? d.Wo : d.W;        // the grid of x
  for (unsigned p = blockIdx.y * 16 + threadIdx.x / kDwV; p < rows; p += gridDim.y * 16) {
    const int j = int(p % Wy), i = int(p / Wy % Hy);
    const bf16* xn = x + int64_t(p / (Wy * Hy)) * Hx * Wx * d.C + c;
    F8 a;
#pragma unroll
    for (int q = 0; q < 8; ++q) a.v[q] = !DGRAD && bias ? bias[c + q] : 0.f;
#pragma unroll
    for (int r = 0; r < KT; ++r) {
      int h = DGRAD ? i + d.pad - r : i * d.stride - d.pad + r;
      bool hok = h >= 0;
      if (DGRAD && d.stride == 2) {
        hok = hok && !(h & 1);
        h >>= 1;
      }
      hok = hok && h < Hx;
      uint4 u[KT];
      bool in[KT];
#pragma unroll
      for (int s = 0; s < KT; ++s) {
        int v = DGRAD ? j + d.pad - s : j * d.stride - d.pad + s;
        bool ok = hok && v >= 0;
        if (DGRAD && d.stride == 2) {
          ok = ok && !(v & 1);
          v >>= 1;
        }
        ok = ok && v < Wx;
        u[s] = *reinterpret_cast<const uint4*>(xn + (ok ? int64_t(h * Wx + v) * d.C : 0));
        in[s] = ok;
      }
#pragma unroll
      for (int s = 0; s < KT; ++s) fma8(a, up8(u[s]), ld8(&ws[r * KT + s][cv]), in[s]);
    }
    bf16* out = y + int64_t(p) * d.C + c;
    if (acc_flag) {
      const F8 o = ld8(out);
#pragma unroll
      for (int q = 0; q < 8; ++q) a.v[q] += o.v[q];
    }
    st8(out, a);
  }
}

// Weight (and bias) gradient partials of pixel chunk blockIdx.y, as
// dwconv_wgrad_k: a thread takes 8 channels and one row of taps, and every
// PL-th pixel of the chunk; the PL pixel lanes are added in order.
template <int KT>
__global__ void __launch_bounds__(240) dwconv_wgrad_x8_k(const bf16* __restrict__ dy, const bf16* __restrict__ x,
                                                         float* __restrict__ pw, float* __restrict__ pb, DwShape d,
                                                         unsigned rows, unsigned per) {
  pdl_wait();
  pdl_trigger();
  constexpr int KK = KT * KT, PL = 240 / (kDwV * KT);
  extern __shared__ float red[];   // [PL][KK + 1][kDwC + 1]
  const int c0 = blockIdx.x * kDwC, nc = min(kDwC, d.C - c0);
  const int cv = 8 * (threadIdx.x % kDwV), c = c0 + cv;
  const int r = threadIdx.x / kDwV % KT, pl = threadIdx.x / (kDwV * KT);
  const unsigned p0 = blockIdx.y * per, p1 = min(rows, p0 + per);
  F8 a[KT], g;
#pragma unroll
  for (int s = 0; s < KT; ++s)
#pragma unroll
    for (int q = 0; q < 8; ++q) a[s].v[q] = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) g.v[q] = 0.f;
  if (cv < nc)
    for (unsigned p = p0 + pl; p < p1; p += PL) {
      const int j = int(p % unsigned(d.Wo)), i = int(p / unsigned(d.Wo) % unsigned(d.Ho));
      const int64_t n = p / (unsigned(d.Wo) * unsigned(d.Ho));
      const int h = i * d.stride - d.pad + r;
      if (r > 0 && (h < 0 || h >= d.H)) continue;
      const F8 dv = ld8(dy + int64_t(p) * d.C + c);
#pragma unroll
      for (int q = 0; q < 8; ++q) g.v[q] += dv.v[q];
      if (h < 0 || h >= d.H) continue;
      const bf16* xr = x + (n * d.H + h) * int64_t(d.W) * d.C + c;
      uint4 u[KT];
      bool in[KT];
#pragma unroll
      for (int s = 0; s < KT; ++s) {   // a tap outside the row loads its first pixel and drops it
        const int v = j * d.stride - d.pad + s;
        in[s] = v >= 0 && v < d.W;
        u[s] = *reinterpret_cast<const uint4*>(xr + (in[s] ? int64_t(v) * d.C : 0));
      }
#pragma unroll
      for (int s = 0; s < KT; ++s) fma8(a[s], dv, up8(u[s]), in[s]);
    }
  float* mine = red + pl * (KK + 1) * (kDwC + 1) + cv;
#pragma unroll
  for (int s = 0; s < KT; ++s)
#pragma unroll
    for (int q = 0; q < 8; ++q) mine[(r * KT + s) * (kDwC + 1) + q] = a[s].v[q];
  if (r == 0)   // row 0 saw every pixel: the bias sum
#pragma unroll
    for (int q = 0; q < 8; ++q) mine[KK * (kDwC + 1) + q] = g.v[q];
  __syncthreads();
  for (int e = threadIdx.x; e < nc * (KK + 1); e += 240) {
    const int cl = e / (KK + 1), t = e % (KK + 1);
    float sum = 0.f;
#pragma unroll
    for (int q = 0; q < PL; ++q) sum += red[(q * (KK + 1) + t) * (kDwC + 1) + cl];
    if (t < KK) pw[int64_t(blockIdx.y) * d.C * KK + int64_t(c0 + cl) * KK + t] = sum;
    else if (pb) pb[int64_t(blockIdx.y) * d.C + c0 + cl] = sum;
  }
}
// 32-bit pixel indices, and 16-byte channel vectors.
bool dw8_ok(const DwShape& d, int dt) {
  return dt == kBF16 && d.C % 8 == 0 && (d.k == 3 || d.k == 5) && int64_t(d.N) * d.H * d.W < (int64_t(1) << 31);
}

int num_sms() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// ------------------------------------------------- hard swish / sigmoid
__device__ __forceinline__ float relu6_p3(float v) { return fminf(fmaxf(v + 3.f, 0.f), 6.f); }

template <typename T>
__global__ void hswish_fwd_k(const T* __restrict__ x, T* __restrict__ y, int64_t n) {
  pdl_wait();
  pdl_trigger();
  FO_MB_GRID_STRIDE(i, n) {
    const float v = to_f(x[i]);
    y[i] = from_f<T>(v * relu6_p3(v) / 6.f);
  }
}
// derivative: 0 below -3, (2x + 3) / 6 on [-3, 3], 1 above 3
template <typename T>
__global__ void hswish_bwd_k(const T* __restrict__ x, const T* __restrict__ dy, T* __restrict__ dx, int64_t n,
                             int acc) {
  pdl_wait();
  pdl_trigger();
  FO_MB_GRID_STRIDE(i, n) {
    const float v = to_f(x[i]);
    const float g = v < -3.f ? 0.f : (v > 3.f ? 1.f : (2.f * v + 3.f) / 6.f);
    store_acc(dx, i, to_f(dy[i]) * g, acc != 0);
  }
}
template <typename T>
__global__ void hsigmoid_fwd_k(const T* __restrict__ x, T* __restrict__ y, int64_t n) {
  pdl_wait();
  pdl_trigger();
  FO_MB_GRID_STRIDE(i, n) y[i] = from_f<T>(relu6_p3(to_f(x[i])) / 6.f);
}
// derivative: 1/6 strictly inside (-3, 3), else 0
template <typename T>
__global__ void hsigmoid_bwd_k(const T* __restrict__ x, const T* __restrict__ dy, T* __restrict__ dx, int64_t n,
                               int acc) {
  pdl_wait();
  pdl_trigger();
  FO_MB_GRID_STRIDE(i, n) {
    const float v = to_f(x[i]);
    store_acc(dx, i, (v > -3.f && v < 3.f) ? to_f(dy[i]) / 6.f : 0.f, acc != 0);
  }
}

// ------------------------------------------------ squeeze-and-excite scale
// y[n,p,c] = x[n,p,c] * s[n,c] over the HW pixels p of image n.
template <typename T>
__global__ void chmul_fwd_k(const T* __restrict__ x, const T* __restrict__ sc, T* __restrict__ y, int N, int HW,
                            int C) {
  pdl_wait();
  pdl_trigger();
  FO_MB_GRID_STRIDE(i, int64_t(N) * HW * C) {
    const int c = int(i % C);
    const int64_t n = i / (int64_t(HW) * C);
    y[i] = from_f<T>(to_f(x[i]) * to_f(sc[n * C + c]));
  }
}
// dx[n,p,c] (+)= dy[n,p,c] s[n,c] (dx may be null);
// ds[n,c] (+)= sum_p dy[n,p,c] x[n,p,c] in pixel order (ds may be null).
template <typename T>
__global__ void chmul_bwd_k(const T* __restrict__ x, const T* __restrict__ sc, const T* __restrict__ dy,
                            T* __restrict__ dx, T* __restrict__ ds, int N, int HW, int C, int acc_dx, int acc_ds) {
  pdl_wait();
  pdl_trigger();
  FO_MB_GRID_STRIDE(o, int64_t(N) * C) {
    const int c = int(o % C);
    const int64_t n = o / C;
    const float s = to_f(sc[o]);
    float sum = 0.f;
    for (int p = 0; p < HW; ++p) {
      const int64_t i = (n * HW + p) * C + c;
      const float g = to_f(dy[i]);
      if (dx) store_acc(dx, i, g * s, acc_dx != 0);
      sum = fmaf(g, to_f(x[i]), sum);
    }
    if (ds) store_acc(ds, o, sum, acc_ds != 0);
  }
}

}  // namespace

void dwconv_fwd(const DwShape& d, const void* x, const void* w, const float* bias, void* y, int dt,
                cudaStream_t st) {
  if (dw8_ok(d, dt)) {
    const unsigned rows = unsigned(d.N) * d.Ho * d.Wo;
    const dim3 grid(ceil_div(d.C, kDwC), std::min(ceil_div(rows, 16), 65535));
    launch_k(d.k == 3 ? dwconv_x8_k<3, false> : dwconv_x8_k<5, false>, grid, kDwThreads, 0, st, (const bf16*)x,
             (const bf16*)w, bias, (bf16*)y, d, rows, 0);
    return;
  }
  const int64_t n = int64_t(d.N) * d.Ho * d.Wo * d.C;
  const int blocks = elementwise_blocks(n, 256);
  FO_MB_DISPATCH(dt, T, {
    if (d.k == 3) launch_k(dwconv_fwd_k<T, 3>, blocks, 256, 0, st, (const T*)x, (const T*)w, bias, (T*)y, d);
    else if (d.k == 5) launch_k(dwconv_fwd_k<T, 5>, blocks, 256, 0, st, (const T*)x, (const T*)w, bias, (T*)y, d);
    else launch_k(dwconv_fwd_k<T, 0>, blocks, 256, 0, st, (const T*)x, (const T*)w, bias, (T*)y, d);
  });
}

void dwconv_dgrad(const DwShape& d, const void* dy, const void* w, void* dx, int dt, bool acc, cudaStream_t st) {
  if (dw8_ok(d, dt)) {
    const unsigned rows = unsigned(d.N) * d.H * d.W;
    const dim3 grid(ceil_div(d.C, kDwC), std::min(ceil_div(rows, 16), 65535));
    launch_k(d.k == 3 ? dwconv_x8_k<3, true> : dwconv_x8_k<5, true>, grid, kDwThreads, 0, st, (const bf16*)dy,
             (const bf16*)w, (const float*)nullptr, (bf16*)dx, d, rows, acc ? 1 : 0);
    return;
  }
  const int64_t n = int64_t(d.N) * d.H * d.W * d.C;
  const int blocks = elementwise_blocks(n, 256);
  const int a = acc ? 1 : 0;
  FO_MB_DISPATCH(dt, T, {
    if (d.k == 3) launch_k(dwconv_dgrad_k<T, 3>, blocks, 256, 0, st, (const T*)dy, (const T*)w, (T*)dx, d, a);
    else if (d.k == 5) launch_k(dwconv_dgrad_k<T, 5>, blocks, 256, 0, st, (const T*)dy, (const T*)w, (T*)dx, d, a);
    else launch_k(dwconv_dgrad_k<T, 0>, blocks, 256, 0, st, (const T*)dy, (const T*)w, (T*)dx, d, a);
  });
}

// Pixel chunks of the weight gradient: for k = 3, 5 about two blocks of 32
// channels per SM, at least 8 pixels (one per warp) per chunk, at most 64
// chunks; for other k, chunks of 32 pixels.
int dwconv_wgrad_chunks(const DwShape& d) {
  const int64_t rows = int64_t(d.N) * d.Ho * d.Wo;
  int64_t q;
  if (d.k == 3 || d.k == 5) {
    const int64_t groups = (d.C + 31) / 32;
    q = (2 * num_sms() + groups - 1) / groups;
    q = std::min<int64_t>(q, (rows + 7) / 8);
  } else {
    q = (rows + 31) / 32;
  }
  q = std::max<int64_t>(1, std::min<int64_t>(q, 64));
  const int64_t per = (rows + q - 1) / q;
  return int((rows + per - 1) / per);
}

void dwconv_wgrad_pass(const DwShape& d, const void* dy, const void* x, int dt, float* pw, float* pb,
                       cudaStream_t st) {
  const int64_t rows = int64_t(d.N) * d.Ho * d.Wo;
  const int chunks = dwconv_wgrad_chunks(d);
  const int per = int((rows + chunks - 1) / chunks);
  if (dw8_ok(d, dt)) {
    const dim3 grid(ceil_div(d.C, kDwC), chunks);
    const size_t sm = sizeof(float) * (240 / (kDwV * d.k)) * (d.k * d.k + 1) * (kDwC + 1);   // below 48 KB
    launch_k(d.k == 3 ? dwconv_wgrad_x8_k<3> : dwconv_wgrad_x8_k<5>, grid, 240, sm, st, (const bf16*)dy,
             (const bf16*)x, pw, pb, d, unsigned(rows), unsigned(per));
    return;
  }
  if (d.k == 3 || d.k == 5) {
    dim3 grid(ceil_div(d.C, 32), chunks);
    FO_MB_DISPATCH(dt, T, {
      if (d.k == 3) launch_k(dwconv_wgrad_k<T, 3>, grid, 256, 0, st, (const T*)dy, (const T*)x, pw, pb, d, per);
      else launch_k(dwconv_wgrad_k<T, 5>, grid, 256, 0, st, (const T*)dy, (const T*)x, pw, pb, d, per);
    });
    return;
  }
  const int taps = d.k * d.k + (pb ? 1 : 0);
  dim3 grid(ceil_div(int64_t(taps) * d.C, 256), chunks);
  FO_MB_DISPATCH(dt, T, launch_k(dwconv_wgrad_any_k<T>, grid, 256, 0, st, (const T*)dy, (const T*)x, pw, pb, d, per));
}

void hswish_fwd(const void* x, void* y, int64_t n, int dt, cudaStream_t st) {
  FO_MB_DISPATCH(dt, T, launch_k(hswish_fwd_k<T>, elementwise_blocks(n, 256), 256, 0, st, (const T*)x, (T*)y, n));
}
void hswish_bwd(const void* x, const void* dy, void* dx, int64_t n, int dt, bool acc, cudaStream_t st) {
  FO_MB_DISPATCH(dt, T, launch_k(hswish_bwd_k<T>, elementwise_blocks(n, 256), 256, 0, st, (const T*)x, (const T*)dy,
                                                                                      (T*)dx, n, acc ? 1 : 0));
}
void hsigmoid_fwd(const void* x, void* y, int64_t n, int dt, cudaStream_t st) {
  FO_MB_DISPATCH(dt, T, launch_k(hsigmoid_fwd_k<T>, elementwise_blocks(n, 256), 256, 0, st, (const T*)x, (T*)y, n));
}
void hsigmoid_bwd(const void* x, const void* dy, void* dx, int64_t n, int dt, bool acc, cudaStream_t st) {
  FO_MB_DISPATCH(dt, T, launch_k(hsigmoid_bwd_k<T>, elementwise_blocks(n, 256), 256, 0, st, (const T*)x, (const T*)dy,
                                                                                        (T*)dx, n, acc ? 1 : 0));
}

void chmul_fwd(const void* x, const void* s, void* y, int N, int HW, int C, int dt, cudaStream_t st) {
  const int64_t n = int64_t(N) * HW * C;
  FO_MB_DISPATCH(dt, T, launch_k(chmul_fwd_k<T>, elementwise_blocks(n, 256), 256, 0, st, (const T*)x, (const T*)s, (T*)y,
                                                                                     N, HW, C));
}
void chmul_bwd(const void* x, const void* s, const void* dy, void* dx, bool acc_dx, void* ds, bool acc_ds, int N,
               int HW, int C, int dt, cudaStream_t st) {
  const int64_t n = int64_t(N) * C;
  FO_MB_DISPATCH(dt, T, launch_k(chmul_bwd_k<T>, elementwise_blocks(n, 256), 256, 0, st, (const T*)x, (const T*)s,
                                                                                     (const T*)dy, (T*)dx, (T*)ds, N,
                                                                                     HW, C, acc_dx ? 1 : 0,
                                                                                     acc_ds ? 1 : 0));
}

}  // namespace fo
