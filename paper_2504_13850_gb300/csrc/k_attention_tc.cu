// Tensor-core multi-head attention for sequences of up to 128 tokens and
// head widths 16, 32, 48 and 64 (bf16 activations): one CTA per (sequence,
// head), the whole 128 x 128 score tile in TMEM.  Same operation as the CUDA-core kernels
// (scaled dot-product attention with keys j >= length[b] masked out):
//   forward   S = Q K^T (TMEM) -> row maximum M of S / sqrt(64) -> P~ =
//             exp(S / 8 - M) (bf16, shared memory) and its row sum ->
//             O = P~ V (TMEM) -> O / row sum (bf16), plus the row
//             log-sum-exp of the scaled scores for the backward pass;
//   backward  S = Q K^T and dP = dO V^T (TMEM) -> P = exp(S / 8 - lse),
//             dS = P (dP - rowsum(dO * O)) / 8 (bf16, shared memory) ->
//             dV = P^T dO, dQ = dS K, dK = dS^T Q (TMEM) -> d(q|k|v).
// (8 stands for the square root of the head width DH.)  Tiles are always 64
// columns wide: a narrower head's tile goes on into its neighbour's columns
// (or zeros past the last), which the products over DH never read and whose
// output columns are not stored.
// Narrower heads keep P and dS in fp32 (SPLIT): a value is multiplied as the
// sum of three bf16 terms, value, remainder and remainder of that, whose 8-bit
// mantissas hold all 24 bits, and each product with a bf16 operand is exact in
// the fp32 accumulator.  The backward then has room for one of P and dS at a
// time: dV = P^T dO first, then dS takes P's tiles.  Two terms (16 bits) were
// not enough: 0.17-0.26% of the outputs and gradients differed from the exact
// value rounded to bf16, against 0.01-0.04% on the fp32 CUDA-core kernels
// that these widths ran on before.  A step of one 256-wide encoder block of
// 19 x 77 tokens, 8 heads of 32: 289 us with those (and the GEMMs of then), 127
// with two terms, 130 with three (64 x 128 tokens: 223 with two, 237 with
// three).
// Operand tiles are 128 rows x 64 bf16 (128-byte rows, 128-byte swizzle),
// loaded by TMA from the packed q|k|v [B*L, 3C] and dO [B*L, C] (the
// backward reads O's rows directly for rowsum(dO * O));
// P (P~ in the forward) and dS are written by the softmax threads in the same swizzled layout as
// two 64-column sub-tiles, which serves both as a K-major operand (P V,
// dS K) and as an MN-major one (P^T dO, dS^T Q).
// Warp roles: warp 0 issues the TMA loads, warp 1 owns TMEM and issues the
// MMAs (one thread each), warps 2..9 do the softmax and the stores: warp w
// reads TMEM lane quarter w % 4 (32 rows) and takes keys 64 * ((w - 2) / 4)
// .. +63 of them, so every row is shared by two threads (the forward pass
// combines their partial maxima and sums through shared memory).  Waits are
// bounded (error word 11..17).
#include "fo_common.cuh"
#include "fo_kernels.h"
#include "fo_ptx.cuh"
#include "fo_tc.h"

namespace fo {

namespace {

constexpr int kAttnThreads = 320;
constexpr int kSoftmaxThreads = 256;      // warps 2..9
constexpr int kTile = 16384;              // 128 rows x 64 bf16

struct AttnParams {
  CUtensorMap tm_qkv;     // [B*L, 3C], box 64 x 128
  CUtensorMap tm_do;      // [B*L, C],  box 64 x 128 (backward)
  const int32_t* len;     // [B]
  const bf16* o;          // backward: the forward output O [B*L, C] (for rowsum(dO * O))
  bf16* out;              // forward: O [B*L, C]; backward: d(q|k|v) [B*L, 3C]
  float* lse;             // [B * heads * L]
  int L, C, heads, acc;
  int* err;
};

// Byte offset of 16-byte unit u (0..7) of row r in a 128-byte-swizzled
// 128 x 64 bf16 tile (8-row groups of 1024 bytes, units XOR-permuted by row).
__device__ __forceinline__ uint32_t sw_off(int r, int u) {
  return uint32_t((r >> 3) * 1024 + (r & 7) * 128 + ((u ^ (r & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Byte offset of term t's tiles from those of term 0 (SPLIT, both passes).
__host__ __device__ constexpr uint32_t term_off(int t) { return t ? uint32_t(2 * t + 1) * kTile : 0u; }

// v[0..8) as a sum of TERMS bf16 values, term t into the 16-byte unit at
// at + term_off(t).  INF: values may be infinite (dS; P is at most 1), and a
// term that is has no remainder.
template <int TERMS, bool INF = false>
__device__ __forceinline__ void st_unit(uint32_t at, float (&v)[8]) {
#pragma unroll
  for (int t = 0; t < TERMS; ++t) {
    uint32_t h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      h[q] = pack_bf16x2(v[2 * q], v[2 * q + 1]);
      if (t + 1 < TERMS) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h[q]));
        v[2 * q] = INF && isinf(f.x) ? 0.f : v[2 * q] - f.x;
        v[2 * q + 1] = INF && isinf(f.y) ? 0.f : v[2 * q + 1] - f.y;
      }
    }
    st_shared4(at + term_off(t), h[0], h[1], h[2], h[3]);
  }
}

template <bool SPLIT>
__device__ __forceinline__ float attn_exp(float x) {
  return SPLIT ? expf(x) : __expf(x);   // the widths that ran in fp32 keep the accurate one
}
template <int DH>
__device__ __forceinline__ float attn_scale() {
  return DH == 64 ? 0.125f : rsqrtf(float(DH));
}

__device__ __forceinline__ char* align1024(char* p) {
  return reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Zeroes the DH columns of row r of a tile, half of them by each thread of the
// row's pair.  A product with a zero P or dS would still be NaN where the other
// operand's row is not finite: SPLIT clears the rows of masked keys and of the
// next sequence, so that whatever those hold stays out, as on the CUDA cores.
template <int DH>
__device__ __forceinline__ void zero_row(const char* tile, int r, int hf) {
#pragma unroll
  for (int u = 0; u < DH / 16; ++u) st_shared4(smem_u32(tile) + sw_off(r, hf * (DH / 16) + u), 0u, 0u, 0u, 0u);
}

// The first N accumulator columns of this lane's row -> N bf16 at dst
// (optionally added to what is there).
template <int N>
__device__ __forceinline__ void store_row(bf16* dst, const uint32_t (&r)[32], bool acc) {
  uint4* d4 = reinterpret_cast<uint4*>(dst);
#pragma unroll
  for (int q = 0; q < N / 8; ++q) {
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[8 * q + e]);
    if (acc) {
      const uint4 o = d4[q];
      const bf16* ob = reinterpret_cast<const bf16*>(&o);
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] += __bfloat162float(ob[e]);
    }
    d4[q] = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                       pack_bf16x2(v[6], v[7]));
  }
}

template <int DH, bool SPLIT>
__global__ void __launch_bounds__(kAttnThreads, 1) attn_fwd_tc_k(const __grid_constant__ AttnParams p) {
  extern __shared__ __align__(1024) char smem_raw[];
  char* sm = align1024(smem_raw);
  char* sQ = sm;
  char* sK = sm + kTile;
  char* sV = sm + 2 * kTile;
  // P~: two sub-tiles (keys 0..63, 64..127); SPLIT: the first term over Q and
  // K, which S = Q K^T alone reads, the others in the tiles after V
  constexpr int kTerms = SPLIT ? 3 : 1;
  char* sP = SPLIT ? sm : sm + 3 * kTile;
  const float kScale = attn_scale<DH>();
  // barriers (ld, s, p, o) and the TMEM slot; SPLIT: as in the backward pass
  uint64_t* bars = reinterpret_cast<uint64_t*>(!SPLIT ? sm + 5 * kTile : (sm - smem_raw >= 64 ? smem_raw : sm + 7 * kTile));
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 4);
  // [half][row]: partial maxima, then sums; SPLIT: in the last unit of V's
  // rows, whose columns no head this narrow has
  auto xch = [&](int half, int row, int sum) -> float* {
    if (SPLIT) return reinterpret_cast<float*>(sV + sw_off(row, 7)) + 2 * sum + half;
    return reinterpret_cast<float*>(sm + 5 * kTile + 64) + (2 * sum + half) * 128 + row;
  };

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int bh = blockIdx.x, b = bh / p.heads, h = bh % p.heads;
  const int row0 = b * p.L;
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    mbar_init(&bars[2], kSoftmaxThreads);
    mbar_init(&bars[3], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&p.tm_qkv)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(256)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;          // S: columns 0..127, O: 128..191
  pdl_trigger();   // this block holds its tensor memory
  pdl_wait();      // the previous kernel's writes are visible from here on

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(&bars[0], 3 * kTile);
      tma_2d(sQ, &p.tm_qkv, &bars[0], h * DH, row0);
      tma_2d(sK, &p.tm_qkv, &bars[0], p.C + h * DH, row0);
      tma_2d(sV, &p.tm_qkv, &bars[0], 2 * p.C + h * DH, row0);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      if (!mbar_wait(&bars[0], 0)) atomicExch(p.err, 11);
      tc_fence_after();
      constexpr uint32_t id_s = instr_desc(128, false, false);
#pragma unroll
      for (int k = 0; k < DH / 16; ++k)
        mma_f16(tmem, smem_desc(smem_u32(sQ) + 32 * k, 16, 1024), smem_desc(smem_u32(sK) + 32 * k, 16, 1024), id_s,
                k > 0 ? 1u : 0u);
      mma_commit(&bars[1]);
      if (!mbar_wait(&bars[2], 0)) atomicExch(p.err, 12);
      tc_fence_after();
      constexpr uint32_t id_o = instr_desc(64, false, true);
#pragma unroll
      for (int t = 0; t < kTerms; ++t)
#pragma unroll
        for (int k = 0; k < 8; ++k)
          mma_f16(tmem + 128, smem_desc(smem_u32(sP) + term_off(t) + (k >> 2) * kTile + 32 * (k & 3), 16, 1024),
                  smem_desc(smem_u32(sV) + 2048 * k, kTile, 1024), id_o, t + k > 0 ? 1u : 0u);
      mma_commit(&bars[3]);
    }
  } else {
    const int q = warp % 4, i = q * 32 + lane, hf = (warp - 2) / 4;
    const uint32_t trow = tmem + (uint32_t(q * 32) << 16) + uint32_t(64 * hf);   // this thread's 64 keys
    const int n = min(p.len[b], p.L);
    if (!mbar_wait(&bars[1], 0)) atomicExch(p.err, 13);
    tc_fence_after();
    // the row maximum over this thread's keys, combined with the other half
    uint32_t r[32];
    float m = -INFINITY;
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      tmem_ld32(trow + 32 * c, r);
      const int j0 = 64 * hf + 32 * c;
#pragma unroll
      for (int e = 0; e < 32; ++e)
        if (j0 + e < n) m = fmaxf(m, __uint_as_float(r[e]) * kScale);
    }
    *xch(hf, i, 0) = m;
    asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
    const float M = fmaxf(m, *xch(1 - hf, i, 0));
    // P~ = exp(s / 8 - M) (bf16, unnormalised: one exponential per score) and
    // its row sum; O = P~ V is normalised by the sum in the store below
    float sum = 0.f;
    const uint32_t p_base = smem_u32(sP) + uint32_t(hf) * kTile;
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      tmem_ld32(trow + 32 * c, r);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int j = 64 * hf + 32 * c + 8 * g + e;
          v[e] = j < n ? attn_exp<SPLIT>(__uint_as_float(r[8 * g + e]) * kScale - M) : 0.f;
          sum += v[e];
        }
        st_unit<kTerms>(p_base + sw_off(i, c * 4 + g), v);
      }
    }
    if (SPLIT && i >= n) zero_row<DH>(sV, i, hf);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // P~ visible to the tensor cores
    tc_fence_before();
    mbar_arrive(&bars[2]);
    // the row sum over both halves, while the tensor cores form O
    *xch(hf, i, 1) = sum;
    asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
    const float S = sum + *xch(1 - hf, i, 1);
    const float inv = S > 0.f ? 1.f / S : 0.f;
    if (hf == 0 && i < p.L) p.lse[size_t(bh) * p.L + i] = M + logf(S);
    if (!mbar_wait(&bars[3], 0)) atomicExch(p.err, 14);
    tc_fence_after();
    // O: DH columns from TMEM column 128 on; each half of the pair stores half of them
    tmem_ld32(tmem + (uint32_t(q * 32) << 16) + 128 + DH / 2 * hf, r);
#pragma unroll
    for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * inv);
    if (i < p.L) store_row<DH / 2>(p.out + size_t(row0 + i) * p.C + h * DH + DH / 2 * hf, r, false);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
  }
}

// Two CTAs per SM: 7 tiles of shared memory (112 KB) and 256 TMEM columns.
// V is read only by the first MMA phase, so P's first sub-tile takes its
// buffer once that phase has completed; O is read from global memory (only
// its row sums with dO are needed); dQ, dV and dK take the TMEM columns of S
// and dP, which the softmax warps have read before the second phase starts.
// SPLIT: 9 tiles, one CTA per SM: the other two terms of P take four more, and
// the terms of dS, held in registers until dV is formed, take those of P.
template <int DH, bool SPLIT>
__global__ void __launch_bounds__(kAttnThreads, SPLIT ? 1 : 2) attn_bwd_tc_k(const __grid_constant__ AttnParams p) {
  extern __shared__ __align__(1024) char smem_raw[];
  char* sm = align1024(smem_raw);
  char* sQ = sm;
  char* sK = sm + kTile;
  char* sV = sm + 2 * kTile;
  char* sP = sm + 2 * kTile;      // two sub-tiles: V's buffer after the first phase, then the next
  char* sdO = sm + 4 * kTile;
  char* sdS = SPLIT ? sP : sm + 5 * kTile;   // two sub-tiles
  constexpr int kTerms = SPLIT ? 3 : 1;
  const float kScale = attn_scale<DH>();
  // barriers (ld, s, p, g and, SPLIT, v: dV formed) and the TMEM slot: in the
  // alignment slack below the tiles when it has room, else after them (the
  // request covers both)
  const bool low = sm - smem_raw >= 64;
  uint64_t* bars = reinterpret_cast<uint64_t*>(low ? smem_raw : sm + (SPLIT ? 9 : 7) * kTile);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 5);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int bh = blockIdx.x, b = bh / p.heads, h = bh % p.heads;
  const int row0 = b * p.L;
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    mbar_init(&bars[2], kSoftmaxThreads);
    mbar_init(&bars[3], 1);
    mbar_init(&bars[4], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&p.tm_qkv)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&p.tm_do)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(256)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // TMEM columns: S 0..127 and dP 128..255; then dQ 0..63, dV 128..191, dK 192..255
  const uint32_t tmem = *tslot;
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(&bars[0], 4 * kTile);
      tma_2d(sQ, &p.tm_qkv, &bars[0], h * DH, row0);
      tma_2d(sK, &p.tm_qkv, &bars[0], p.C + h * DH, row0);
      tma_2d(sV, &p.tm_qkv, &bars[0], 2 * p.C + h * DH, row0);
      tma_2d(sdO, &p.tm_do, &bars[0], h * DH, row0);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      if (!mbar_wait(&bars[0], 0)) atomicExch(p.err, 15);
      tc_fence_after();
      constexpr uint32_t id_nn128 = instr_desc(128, false, false);
#pragma unroll
      for (int k = 0; k < DH / 16; ++k) {
        mma_f16(tmem, smem_desc(smem_u32(sQ) + 32 * k, 16, 1024), smem_desc(smem_u32(sK) + 32 * k, 16, 1024),
                id_nn128, k > 0 ? 1u : 0u);
        mma_f16(tmem + 128, smem_desc(smem_u32(sdO) + 32 * k, 16, 1024),
                smem_desc(smem_u32(sV) + 32 * k, 16, 1024), id_nn128, k > 0 ? 1u : 0u);
      }
      mma_commit(&bars[1]);
      if (!mbar_wait(&bars[2], 0)) atomicExch(p.err, 16);
      tc_fence_after();
      constexpr uint32_t id_tt = instr_desc(64, true, true);    // dV, dK: A and B MN-major
      constexpr uint32_t id_nt = instr_desc(64, false, true);   // dQ: A K-major, B MN-major
      // dV[j][d] = sum_i P[i][j] dO[i][d]
      auto dv_mma = [&](int t, int k) {
        mma_f16(tmem + 128, smem_desc(smem_u32(sP) + term_off(t) + 2048 * k, kTile, 1024),
                smem_desc(smem_u32(sdO) + 2048 * k, kTile, 1024), id_tt, t + k > 0 ? 1u : 0u);
      };
      // dQ[i][d] = sum_j dS[i][j] K[j][d] and dK[j][d] = sum_i dS[i][j] Q[i][d]
      auto dqk_mma = [&](int t, int k) {
        const uint32_t ds = smem_u32(sdS) + term_off(t), acc = t + k > 0 ? 1u : 0u;
        mma_f16(tmem, smem_desc(ds + (k >> 2) * kTile + 32 * (k & 3), 16, 1024),
                smem_desc(smem_u32(sK) + 2048 * k, kTile, 1024), id_nt, acc);
        mma_f16(tmem + 192, smem_desc(ds + 2048 * k, kTile, 1024), smem_desc(smem_u32(sQ) + 2048 * k, kTile, 1024),
                id_tt, acc);
      };
      if constexpr (SPLIT) {
#pragma unroll
        for (int t = 0; t < kTerms; ++t)
#pragma unroll
          for (int k = 0; k < 8; ++k) dv_mma(t, k);
        mma_commit(&bars[4]);
        if (!mbar_wait(&bars[2], 1)) atomicExch(p.err, 16);   // dS in P's place
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < kTerms; ++t)
#pragma unroll
          for (int k = 0; k < 8; ++k) dqk_mma(t, k);
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          dv_mma(0, k);
          dqk_mma(0, k);
        }
      }
      mma_commit(&bars[3]);
    }
  } else {
    const int q = warp % 4, i = q * 32 + lane, hf = (warp - 2) / 4;   // keys 64 hf .. +63
    const uint32_t trow = tmem + (uint32_t(q * 32) << 16);
    const int n = min(p.len[b], p.L);
    const bool live = i < p.L;          // rows past the sequence get P = dS = 0
    // D_i = sum_d dO[i][d] O[i][d]: O's row from global memory (in flight
    // during the TMA wait), dO's from the swizzled tile
    uint4 orow[DH / 8];
#pragma unroll
    for (int u = 0; u < DH / 8; ++u) orow[u] = make_uint4(0u, 0u, 0u, 0u);
    if (live) {
      const uint4* src = reinterpret_cast<const uint4*>(p.o + size_t(row0 + i) * p.C + h * DH);
#pragma unroll
      for (int u = 0; u < DH / 8; ++u) orow[u] = src[u];
    }
    if (!mbar_wait(&bars[0], 0)) atomicExch(p.err, 15);
    float D = 0.f;
    const uint32_t do_base = smem_u32(sdO);
#pragma unroll
    for (int u = 0; u < DH / 8; ++u) {
      const float4 a = ld_shared4(do_base + sw_off(i, u));
      const bf16* ab = reinterpret_cast<const bf16*>(&a);
      const bf16* cb = reinterpret_cast<const bf16*>(&orow[u]);
#pragma unroll
      for (int e = 0; e < 8; ++e) D = fmaf(__bfloat162float(ab[e]), __bfloat162float(cb[e]), D);
    }
    const float lse = live ? p.lse[size_t(bh) * p.L + i] : 0.f;
    if (!mbar_wait(&bars[1], 0)) atomicExch(p.err, 13);
    tc_fence_after();
    const uint32_t p_base = smem_u32(sP), ds_base = smem_u32(sdS);
    // scores 32 cc .. +31 of this thread's 64: P into its tile, dS into its own
    // or (SPLIT) `ds`
    auto chunk = [&](int cc, float* ds) {
      const int c = 2 * hf + cc;
      uint32_t rs[32], rp[32];
      tmem_ld32(trow + 32 * c, rs);
      tmem_ld32(trow + 128 + 32 * c, rp);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float pv[8], dv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int j = 32 * c + 8 * g + e;
          const bool in = live && j < n;
          const float pj = in ? attn_exp<SPLIT>(__uint_as_float(rs[8 * g + e]) * kScale - lse) : 0.f;
          pv[e] = pj;
          dv[e] = pj * (__uint_as_float(rp[8 * g + e]) - D) * kScale;
          if (SPLIT && !in) dv[e] = 0.f;
          if (SPLIT) ds[32 * cc + 8 * g + e] = dv[e];
        }
        const uint32_t off = (c >> 1) * kTile + sw_off(i, (c & 1) * 4 + g);
        st_unit<kTerms>(p_base + off, pv);
        if (!SPLIT) st_unit<1>(ds_base + off, dv);
      }
    };
    auto release = [&] {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // P, dS visible to the tensor cores
      tc_fence_before();
      mbar_arrive(&bars[2]);
    };
    if constexpr (SPLIT) {
      float ds[64];
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) chunk(cc, ds);
      if (i >= n) zero_row<DH>(sK, i, hf);
      if (!live) {
        zero_row<DH>(sQ, i, hf);
        zero_row<DH>(sdO, i, hf);
      }
      release();
      if (!mbar_wait(&bars[4], 0)) atomicExch(p.err, 17);   // P's tiles are free
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = ds[8 * u + e];
        st_unit<kTerms, true>(ds_base + hf * kTile + sw_off(i, u), v);
      }
    } else {
#pragma unroll 1
      for (int cc = 0; cc < 2; ++cc) chunk(cc, nullptr);
    }
    release();
    if (!mbar_wait(&bars[3], 0)) atomicExch(p.err, 14);
    tc_fence_after();
    // TMEM row i holds dQ row i and dK / dV row j = i; each half of the
    // pair stores half of the DH columns of each
    bf16* drow = p.out + size_t(row0 + i) * 3 * p.C;
#pragma unroll 1
    for (int t = 0; t < 3; ++t) {
      const uint32_t col = t == 0 ? 0u : (t == 1 ? 192u : 128u);     // dQ, dK, dV
      uint32_t r[32];
      tmem_ld32(trow + col + DH / 2 * hf, r);
      if (SPLIT && t > 0 && i >= n)
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = 0u;   // no gradient of a masked key
      if (live) store_row<DH / 2>(drow + t * p.C + h * DH + DH / 2 * hf, r, p.acc != 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
  }
}

constexpr size_t kFwdSmem = 5 * kTile + 1024 + 64 + 4 * 128 * sizeof(float2);
constexpr size_t kBwdSmem = 7 * kTile + 1024;   // 115,712 B: two CTAs in an SM's 228 KB
constexpr size_t kFwdSplitSmem = 7 * kTile + 1024;   // two CTAs as well
constexpr size_t kBwdSplitSmem = 9 * kTile + 1024;

typedef void (*AttnKernel)(const AttnParams);
struct AttnKernels {
  AttnKernel fwd, bwd;
  size_t fwd_smem, bwd_smem;
};
// The kernels of a head width, or nulls.
AttnKernels attn_kernels(int dh) {
  switch (dh) {
    case 16: return {attn_fwd_tc_k<16, true>, attn_bwd_tc_k<16, true>, kFwdSplitSmem, kBwdSplitSmem};
    case 32: return {attn_fwd_tc_k<32, true>, attn_bwd_tc_k<32, true>, kFwdSplitSmem, kBwdSplitSmem};
    case 48: return {attn_fwd_tc_k<48, true>, attn_bwd_tc_k<48, true>, kFwdSplitSmem, kBwdSplitSmem};
    case 64: return {attn_fwd_tc_k<64, false>, attn_bwd_tc_k<64, false>, kFwdSmem, kBwdSmem};
  }
  return {nullptr, nullptr, 0, 0};
}

}  // namespace

struct AttnTcPlan {
  AttnParams p;
  AttnKernels k;
};

// Head widths that are multiples of the MMA's K of 16 (so every box also
// starts on a 16-byte boundary); others stay on the CUDA cores.
bool attention_tc_ok(int L, int C, int heads) {
  return L >= 1 && L <= 128 && heads > 0 && C % heads == 0 && attn_kernels(C / heads).fwd != nullptr;
}

AttnTcPlan* attention_tc_plan(const void* qkv, const void* out, const void* dout, int B, int L, int C, int heads,
                              int* err) {
  if (!attention_tc_ok(L, C, heads)) return nullptr;
  AttnTcPlan* a = new AttnTcPlan();
  a->p = AttnParams{};
  a->k = attn_kernels(C / heads);
  a->p.L = L;
  a->p.C = C;
  a->p.heads = heads;
  a->p.err = err;
  a->p.o = static_cast<const bf16*>(out);
  const int64_t rows = int64_t(B) * L;
  if (!tc_encode_2d(&a->p.tm_qkv, qkv, rows, 3 * C, 128) ||
      (dout && !tc_encode_2d(&a->p.tm_do, dout, rows, C, 128))) {
    delete a;
    return nullptr;
  }
  // Sized for two CTAs per SM (the backward of the narrower heads for one),
  // which needs the largest shared-memory carveout (the default sizes the
  // carveout for one block).
  const int most = int(cudaSharedmemCarveoutMaxShared);
  if (cudaFuncSetAttribute(a->k.fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, int(a->k.fwd_smem)) != cudaSuccess ||
      cudaFuncSetAttribute(a->k.bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, int(a->k.bwd_smem)) != cudaSuccess ||
      cudaFuncSetAttribute(a->k.fwd, cudaFuncAttributePreferredSharedMemoryCarveout, most) != cudaSuccess ||
      cudaFuncSetAttribute(a->k.bwd, cudaFuncAttributePreferredSharedMemoryCarveout, most) != cudaSuccess) {
    delete a;
    return nullptr;
  }
  return a;
}

void attention_tc_destroy(AttnTcPlan* a) { delete a; }

void attention_tc_fwd(const AttnTcPlan* a, const int32_t* len, void* out, float* lse, int B, cudaStream_t st) {
  AttnParams p = a->p;
  p.len = len;
  p.out = static_cast<bf16*>(out);
  p.lse = lse;
  p.acc = 0;
  launch_k(a->k.fwd, B * p.heads, kAttnThreads, a->k.fwd_smem, st, p);
}

void attention_tc_bwd(const AttnTcPlan* a, const int32_t* len, const float* lse, void* dqkv, int B, bool acc,
                      cudaStream_t st) {
  AttnParams p = a->p;
  p.len = len;
  p.out = static_cast<bf16*>(dqkv);
  p.lse = const_cast<float*>(lse);
  p.acc = acc ? 1 : 0;
  launch_k(a->k.bwd, B * p.heads, kAttnThreads, a->k.bwd_smem, st, p);
}

}  // namespace fo
