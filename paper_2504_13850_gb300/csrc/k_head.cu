// Classifier head of the server network: the last linear layer (few
// outputs) fused with the server loss f_s (softmax cross-entropy averaged
// over the batch) and its backward pass.
//   head_fwd_ce : logits z = x W^T + b, per-row CE, dz = (softmax(z) - onehot)/B,
//                 and (optionally, in the same launch) dx (+)= dz W, times a
//                 ReLU mask (mask > 0) when one is given
//   head_wgrad  : dW = dz^T x, db = sum_b dz, loss = mean of the row losses
//                 (summed in row order, deterministic)
// W and b are the fp32 master weights; dz and the gradients are fp32.
#include "fo_common.cuh"
#include "fo_kernels.h"

#include <algorithm>
#include <type_traits>

namespace fo {

namespace {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// V consecutive elements (V = 4: the address is a multiple of four elements).
template <int V>
__device__ __forceinline__ void ldv(const float* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const float4 f = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
  } else {
    v[0] = *p;
  }
}
template <int V>
__device__ __forceinline__ void ldv(const bf16* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    const bf16* e = reinterpret_cast<const bf16*>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __bfloat162float(e[i]);
  } else {
    v[0] = __bfloat162float(*p);
  }
}

// Sums v[0..N) over the warp's lanes (N a power of two <= 32) by halving the
// values a lane carries at each exchange: lane l ends with the sum of value
// l >> (5 - log2 N) in v[0].
template <int N>
__device__ __forceinline__ void lanes_sum(float (&v)[N], int lane) {
  int off = 16;
#pragma unroll
  for (int n = N; n > 1; n /= 2, off /= 2) {
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float keep = hi ? v[i + n / 2] : v[i], send = hi ? v[i] : v[i + n / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (; off > 0; off /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}

constexpr int kHeadCtas = 8;      // CTAs of a cluster
constexpr int kHeadThreads = 256;

__device__ __forceinline__ float ld_peer(const float* p, uint32_t rank) {
  uint32_t a = uint32_t(__cvta_generic_to_shared(p)), r;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r) : "memory");
  return v;
}

// A cluster of eight CTAs takes R batch rows: each CTA forms the logits of an
// eighth of the classes (a warp: four classes of all R rows, the contraction
// split over the warps that few classes leave over), all gather the R x C
// logits through distributed shared memory and form the softmax and dz, and
// each CTA forms an eighth of the rows' input gradient
//   dx[b][k] (+)= (sum_c dz[b][c] W[c][k]) * (mask[b][k] > 0)   (if dx is given).
// What bounds it is reading W (fp32, from L2): one block per row read all of
// it twice by itself, at the rate of one SM; here a CTA reads a quarter of W
// for its R rows, with four-wide loads where K allows (V = 4).
// Launch alone, us, one block per row -> here: 64 rows x 1280 -> 200 classes
// 85.5 -> 27.4; 16 x 4096 -> 10 (fp32) 30.9 -> 9.2.  Steps: MobileNet 476 -> 417,
// ResNet on 28 x 28 maps with 1000 classes 654 -> 515, tiny fp32 95 -> 81.
template <typename T, int R, int V>
__global__ void __launch_bounds__(kHeadThreads) head_fwd_ce_k(
    const T* __restrict__ x, const float* __restrict__ W, const float* __restrict__ bias,
    const int32_t* __restrict__ labels, int B, int K, int C, float* __restrict__ logits, float* __restrict__ dz,
    float* __restrict__ row_loss, const T* __restrict__ mask, T* __restrict__ dx, int acc) {
  extern __shared__ __align__(16) float sm[];
  const int per = (C + kHeadCtas - 1) / kHeadCtas;   // classes per CTA
  float* z = sm;                                     // [R][C]: logits, then dz
  float* zs = z + R * C;                             // [R][per]: this CTA's logits
  float* part = zs + R * per;                        // partial sums of both products
  const uint32_t rank = blockIdx.x % kHeadCtas;
  const int b0 = int(blockIdx.x / kHeadCtas) * R, rows = min(R, B - b0);
  const int c0 = min(C, int(rank) * per), c1 = min(C, c0 + per);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  pdl_wait();
  pdl_trigger();

  // logits of classes c0 .. c1 - 1: `gw` warps over groups of four classes,
  // the contraction split over 8 / gw warps
  const int groups = (per + 3) / 4;
  int gw = 1;
  while (gw < groups && gw < 8) gw *= 2;
  const int splits = 8 / gw, kw = warp / gw;
  for (int g = warp % gw; g < groups; g += gw) {
    const float* w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = W + int64_t(min(c0 + 4 * g + j, C - 1)) * K;
    float s[4 * R];
#pragma unroll
    for (int e = 0; e < 4 * R; ++e) s[e] = 0.f;
#pragma unroll 2
    for (int k = (kw * 32 + lane) * V; k < K; k += splits * 32 * V) {
      float wv[4][V];
#pragma unroll
      for (int j = 0; j < 4; ++j) ldv<V>(w[j] + k, wv[j]);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float xv[V];
        ldv<V>(x + int64_t(b0 + min(r, rows - 1)) * K + k, xv);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int v = 0; v < V; ++v) s[j * R + r] = fmaf(xv[v], wv[j][v], s[j * R + r]);
      }
    }
    lanes_sum<4 * R>(s, lane);
    const int e = lane / (32 / (4 * R)), c = 4 * g + e / R;
    if (lane % (32 / (4 * R)) == 0 && c < per) part[(kw * R + e % R) * per + c] = s[0];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < R * per; e += kHeadThreads) {
    float s = 0.f;
    for (int q = 0; q < splits; ++q) s += part[q * R * per + e];
    const int c = c0 + e % per;
    zs[e] = s + (bias && c < C ? bias[c] : 0.f);
  }
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  for (int e = threadIdx.x; e < R * C; e += kHeadThreads) {
    const int r = e / C, c = e % C;
    z[e] = ld_peer(zs + r * per + c % per, uint32_t(c / per));
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");   // this CTA's reads of its peers are done
  __syncthreads();

  if (warp < R) {   // one warp per row: softmax cross-entropy and dz
    float* zr = z + warp * C;
    float m = -INFINITY;
    for (int c = lane; c < C; c += 32) m = fmaxf(m, zr[c]);
    m = warp_max(m);
    float se = 0.f;
    for (int c = lane; c < C; c += 32) se += expf(zr[c] - m);
    se = warp_sum(se);
    const int b = b0 + warp;
    const bool live = warp < rows;
    const int y = live ? labels[b] : -1;
    if (live && rank == 0 && lane == 0) row_loss[b] = m + logf(se) - (y >= 0 && y < C ? zr[y] : 0.f);
    __syncwarp();
    for (int c = lane; c < C; c += 32) {
      const float v = zr[c], p = expf(v - m) / se;
      const float d = live ? (p - (c == y ? 1.f : 0.f)) / float(B) : 0.f;
      if (live && c >= c0 && c < c1) {
        dz[int64_t(b) * C + c] = d;
        logits[int64_t(b) * C + c] = v;
      }
      zr[c] = d;
    }
  }
  __syncthreads();

  if (dx) {
    const int vecs = K / V, pv = (vecs + kHeadCtas - 1) / kHeadCtas;   // V-wide columns, per CTA
    const int v0 = min(vecs, int(rank) * pv), v1 = min(vecs, v0 + pv);
    int tc = 8;                                    // threads over columns; the rest split the classes
    while (tc < pv && tc < kHeadThreads) tc *= 2;
    const int cs = kHeadThreads / tc, col = threadIdx.x % tc, cq = threadIdx.x / tc;
    for (int vb = v0; vb < v1; vb += tc) {
      float s[R][V];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) s[r][v] = 0.f;
      if (vb + col < v1) {
#pragma unroll 4
        for (int c = cq; c < C; c += cs) {
          float wv[V];
          ldv<V>(W + int64_t(c) * K + int64_t(vb + col) * V, wv);
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const float d = z[r * C + c];
#pragma unroll
            for (int v = 0; v < V; ++v) s[r][v] = fmaf(d, wv[v], s[r][v]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) part[(cq * R + r) * tc * V + col * V + v] = s[r][v];
      __syncthreads();
      const int width = min(tc, v1 - vb) * V;
      for (int e = threadIdx.x; e < rows * tc * V; e += kHeadThreads) {
        const int r = e / (tc * V), k = e % (tc * V);
        if (k >= width) continue;
        float t = 0.f;
        for (int q = 0; q < cs; ++q) t += part[q * R * tc * V + e];
        const int64_t i = int64_t(b0 + r) * K + int64_t(vb) * V + k;
        if (mask && !(to_f(mask[i]) > 0.f)) t = 0.f;
        if (acc) t += to_f(dx[i]);
        dx[i] = from_f<T>(t);
      }
      __syncthreads();
    }
  }
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // no peer still reads this CTA's logits
}

// dW[c][k] = sum_b dz[b][c] x[b][k]: block = 32 columns k x 8 classes c,
// rows staged through shared memory 64 at a time; grid (ceil(K/32),
// ceil(C/8)).  Block (0, y) also writes db for its classes; block (0, 0)
// the batch-mean loss (row order).
template <typename T>
__global__ void head_wgrad_k(const float* __restrict__ dz, const T* __restrict__ x, int B, int K, int C,
                             float* __restrict__ dW, float* __restrict__ db, const float* __restrict__ row_loss,
                             float* __restrict__ losses, const int64_t* __restrict__ step, int64_t mask,
                             float* __restrict__ mirror, int64_t mirror_mask) {
  pdl_wait();
  pdl_trigger();
  __shared__ float xs[64][33];
  __shared__ float ds[64][8];
  __shared__ float rl[1024];   // the row losses (a batch has at most 1024 rows)
  const int kk = threadIdx.x % 32, cc = threadIdx.x / 32;
  const int k = blockIdx.x * 32 + kk, c = blockIdx.y * 8 + cc;
  float acc = 0.f, dsum = 0.f;
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int b = threadIdx.x; b < B; b += blockDim.x) rl[b] = row_loss[b];
  for (int b0 = 0; b0 < B; b0 += 64) {
    for (int e = threadIdx.x; e < 64 * 32; e += blockDim.x) {
      const int b = b0 + e / 32, kx = blockIdx.x * 32 + e % 32;
      xs[e / 32][e % 32] = (b < B && kx < K) ? to_f(x[int64_t(b) * K + kx]) : 0.f;
    }
    for (int e = threadIdx.x; e < 64 * 8; e += blockDim.x) {
      const int b = b0 + e / 8, cx = blockIdx.y * 8 + e % 8;
      ds[e / 8][e % 8] = (b < B && cx < C) ? dz[int64_t(b) * C + cx] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int b = 0; b < 64; ++b) acc = fmaf(ds[b][cc], xs[b][kk], acc);
    if (blockIdx.x == 0)   // rows past B are zeros
#pragma unroll 8
      for (int b = 0; b < 64; ++b) dsum += ds[b][cc];
    __syncthreads();
  }
  if (k < K && c < C) dW[int64_t(c) * K + k] = acc;
  if (blockIdx.x == 0 && kk == 0 && c < C) {
    if (db) db[c] = dsum;
    if (c == 0) {
      float t = 0.f;
#pragma unroll 8
      for (int b = 0; b < B; ++b) t += rl[b];
      losses[*step & mask] = t / float(B);
      if (mirror) mirror[*step & mirror_mask] = t / float(B);
    }
  }
}

// Floats of the head's shared memory: logits of R rows, this CTA's share of
// them, and the partial sums of both products: of the logits R x per x (8 /
// warps over class groups), at most R x max(per, 32), and of dx R x 256 V.
size_t head_floats(int R, int V, int C) {
  const int per = (C + kHeadCtas - 1) / kHeadCtas;
  return size_t(R) * (size_t(C) + per + std::max(kHeadThreads * V, std::max(per, 32)));
}
constexpr int kHeadMaxClasses = 1024;   // more classes take the unfused loss

}  // namespace

void head_forward_loss(const void* x, int dt, const float* W, const float* bias, const int32_t* labels, int B,
                       int K, int C, float* logits, float* dz, float* row_loss, cudaStream_t st, const void* mask,
                       void* dx, bool acc) {
  // rows per cluster: the fewest that need at most 16 clusters (128 CTAs), up to 8
  int R = 1;
  while (R < 8 && (B + R - 1) / R > 16) R *= 2;
  const int V = K % 4 == 0 ? 4 : 1;   // rows of W and x stay aligned
  const size_t sm = sizeof(float) * head_floats(R, V, C);
  auto go = [&](auto kernel, auto tag) {
    typedef decltype(tag) T;
    // the same limit in every call: servers of other class counts may launch from other threads meanwhile
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         int(sizeof(float) * head_floats(R, V, kHeadMaxClasses)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned((B + R - 1) / R) * kHeadCtas);
    cfg.blockDim = dim3(kHeadThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kHeadCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, (const T*)x, W, bias, labels, B, K, C, logits, dz, row_loss, (const T*)mask,
                       (T*)dx, acc ? 1 : 0);
  };
  auto rows = [&](auto tag, auto vec) {
    typedef decltype(tag) T;
    constexpr int VV = decltype(vec)::value;
    if (R == 1) go(head_fwd_ce_k<T, 1, VV>, tag);
    else if (R == 2) go(head_fwd_ce_k<T, 2, VV>, tag);
    else if (R == 4) go(head_fwd_ce_k<T, 4, VV>, tag);
    else go(head_fwd_ce_k<T, 8, VV>, tag);
  };
  auto type = [&](auto vec) {
    if (dt == kF32) rows(float(), vec);
    else rows(bf16(), vec);
  };
  if (V == 4) type(std::integral_constant<int, 4>());
  else type(std::integral_constant<int, 1>());
}

void head_weight_grad(const float* dz, const void* x, int dt, int B, int K, int C, float* dW, float* db,
                      const float* row_loss, float* losses, const int64_t* step, int64_t mask,
                      cudaStream_t st, float* mirror, int64_t mirror_mask) {
  dim3 grid(ceil_div(K, 32), ceil_div(C, 8));
  if (dt == kF32)
    launch_k(head_wgrad_k<float>, grid, 256, 0, st, dz, (const float*)x, B, K, C, dW, db, row_loss, losses, step, mask, mirror,
             mirror_mask);
  else
    launch_k(head_wgrad_k<bf16>, grid, 256, 0, st, dz, (const bf16*)x, B, K, C, dW, db, row_loss, losses, step, mask, mirror,
             mirror_mask);
}

}  // namespace fo
