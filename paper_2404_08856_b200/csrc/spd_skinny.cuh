// Y[M,N] = X[M,K] W[N,K]^T for M <= 8 on weights as the caller has them (row-major): the stand-alone form
// of the verify projections.  HBM-bound: every weight is read once, straight into registers, and used
// there; nothing is repacked.  (Repacking into the streaming layout of the forward kernel and running
// its projection on the copy moved every weight three times: 12288 x 4096 bf16, M = 6: 96 us, this way
// 25 us = 4.0 TB/s; 688 x 256 fp32, M = 4: 13.6 -> 6.1 us.)
//
// A CTA of 16 warps on every SM; a group of KS warps shares a run of rows and splits K, so that a warp
// has a few hundred bytes of every row; their partial sums meet in shared memory once per tile, one
// barrier, two buffers.  A warp requests the next tile's weights before the current tile's sums are
// exchanged, and the first tile's before the activations are prepared.  Rows are dealt evenly to all
// groups: a small N gives every group one or no row.
//  * bf16: mma.m16n8k16 with 16 weight rows as the A operand, loaded as 16-byte pieces (the K order
//    inside a 32-wide block is whatever the loads give, the activations are laid out to match), the
//    activations as bf16 hi + lo B fragments in shared memory.
//  * fp32: 4 rows per tile, lanes split K, packed fp32 FMAs, butterfly over the lanes.
#pragma once
#include "spd_engine.cuh"

namespace spd {

constexpr int SK_WARPS = 16, SK_THREADS = SK_WARPS * 32;
constexpr int SK_RED = 2 * SK_WARPS * 128 * 4;            // two buffers of 128 partial sums per warp
constexpr int SK_X_MAX = 192 * 1024;                      // activations resident in shared memory
constexpr int SK_BLOCKS = 8;                              // bf16: 32-wide K blocks of a tile in flight per warp
constexpr int SK_BLOCKS_F32 = 2;                          // fp32: 128-wide

__host__ __device__ constexpr int sk_kb(int K, int esz) { return esz == 2 ? (K + 31) / 32 : (K + 127) / 128; }
// bytes of the prepared activations
__host__ __device__ constexpr long long sk_x_bytes(int M, int K, int esz) {
  return esz == 2 ? (long long)sk_kb(K, 2) * 1024 : (long long)M * sk_kb(K, 4) * 512;
}

// The partial sums of a tile: `cnt` values per warp in `red`, summed over the KS warps of the group in
// order; value i goes to out(i, sum).
template <class OUT>
__device__ __forceinline__ void sk_exchange(const float* red, int group, int KS, int cnt, OUT out) {
  if (KS > 1) named_sync(1 + group, KS * 32);
  else __syncwarp();
  const int t = threadIdx.x - group * KS * 32;
  for (int i = t; i < cnt; i += KS * 32) {
    float v = 0.f;
    for (int w = 0; w < KS; ++w) v += red[(group * KS + w) * 128 + i];
    out(i, v);
  }
}

__global__ void __launch_bounds__(SK_THREADS, 1)
skinny_bf16_kernel(const float* x, const __nv_bfloat16* w, int M, int N, int K, float* y, int KS, int* clear) {
  extern __shared__ __align__(1024) char sk_sm[];
  float* red = reinterpret_cast<float*>(sk_sm);
  uint4* frag = reinterpret_cast<uint4*>(sk_sm + SK_RED);          // [KB][2][32]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
  if (clear && blockIdx.x == 0 && tid == 0) *clear = 0;
  const int KB = sk_kb(K, 2), groups = SK_WARPS / KS, group = warp / KS, slice = warp - group * KS;
  const long long G = (long long)gridDim.x * groups, gi = (long long)group * gridDim.x + blockIdx.x;
  const int r0 = (int)(N * gi / G), r1 = (int)(N * (gi + 1) / G);
  const int per = (KB + KS - 1) / KS, b0 = min(KB, slice * per), b1 = min(KB, b0 + per);
  const int batches = (per + SK_BLOCKS - 1) / SK_BLOCKS;
  const int tiles = (r1 - r0 + 15) / 16, steps = tiles * batches;

  uint4 a[SK_BLOCKS][2];
  auto load = [&](int step) {
    const int row = r0 + (step / batches) * 16 + gq, kb = b0 + (step % batches) * SK_BLOCKS;
#pragma unroll
    for (int i = 0; i < SK_BLOCKS; ++i) {
      const int k = (kb + i) * 32 + tq * 8;
      const bool in = kb + i < b1 && k < K;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        a[i][h] = in && row + 8 * h < r1 ? __ldcs(reinterpret_cast<const uint4*>(w + (size_t)(row + 8 * h) * K + k))
                                         : make_uint4(0, 0, 0, 0);
    }
  };
  if (steps > 0) load(0);
  // activations -> B fragments: block kb, step s, lane (m = gq, k = kb * 32 + tq * 8 + 4 s ..): hi pair, hi pair, lo, lo
  for (int i = tid; i < KB * 64; i += SK_THREADS) {
    const int l = i & 31, s = (i >> 5) & 1, kb = i >> 6, m = l >> 2, k = kb * 32 + (l & 3) * 8 + 4 * s;
    const float4 v = m < M && k < K ? __ldg(reinterpret_cast<const float4*>(x + (size_t)m * K + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    uint4 f;
    f.x = pack_bf16(v.x, v.y);
    f.y = pack_bf16(v.z, v.w);
    f.z = pack_bf16(v.x - bf16lo(f.x), v.y - bf16hi(f.x));
    f.w = pack_bf16(v.z - bf16lo(f.y), v.w - bf16hi(f.y));
    frag[i] = f;
  }
  __syncthreads();
  float hi[4], lo[4];
  for (int step = 0; step < steps; ++step) {
    const int t = step / batches, bt = step - t * batches, kb = b0 + bt * SK_BLOCKS;
    if (bt == 0)
#pragma unroll
      for (int j = 0; j < 4; ++j) hi[j] = lo[j] = 0.f;
#pragma unroll
    for (int i = 0; i < SK_BLOCKS; ++i) {
      if (kb + i >= b1) break;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const uint4 f = frag[((kb + i) * 2 + s) * 32 + lane];
        const uint32_t a0 = s ? a[i][0].z : a[i][0].x, a2 = s ? a[i][0].w : a[i][0].y;
        const uint32_t a1 = s ? a[i][1].z : a[i][1].x, a3 = s ? a[i][1].w : a[i][1].y;
        mma_bf16(hi, a0, a1, a2, a3, f.x, f.y);
        mma_bf16(lo, a0, a1, a2, a3, f.z, f.w);
      }
    }
    if (step + 1 < steps) load(step + 1);
    if (bt + 1 == batches) {
      float* mine = red + (t & 1) * SK_WARPS * 128;
      *reinterpret_cast<float2*>(mine + warp * 128 + gq * 8 + tq * 2) = make_float2(hi[0] + lo[0], hi[1] + lo[1]);
      *reinterpret_cast<float2*>(mine + warp * 128 + (gq + 8) * 8 + tq * 2) = make_float2(hi[2] + lo[2], hi[3] + lo[3]);
      const int row0 = r0 + t * 16;
      sk_exchange(mine, group, KS, 128, [&](int i, float v) {
        const int row = row0 + (i >> 3), m = i & 7;
        if (row < r1 && m < M) y[(size_t)m * N + row] = v;
      });
    }
  }
}

template <int M>
__global__ void __launch_bounds__(SK_THREADS, 1)
skinny_f32_kernel(const float* x, const float* w, int N, int K, float* y, int KS, int* clear) {
  extern __shared__ __align__(1024) char sk_sm[];
  float* red = reinterpret_cast<float*>(sk_sm);
  float* xs = reinterpret_cast<float*>(sk_sm + SK_RED);             // [M][KB * 128]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (clear && blockIdx.x == 0 && tid == 0) *clear = 0;
  const int KB = sk_kb(K, 4), groups = SK_WARPS / KS, group = warp / KS, slice = warp - group * KS;
  const long long G = (long long)gridDim.x * groups, gi = (long long)group * gridDim.x + blockIdx.x;
  const int r0 = (int)(N * gi / G), r1 = (int)(N * (gi + 1) / G);
  const int per = (KB + KS - 1) / KS, b0 = min(KB, slice * per), b1 = min(KB, b0 + per);
  const int batches = (per + SK_BLOCKS_F32 - 1) / SK_BLOCKS_F32;
  const int tiles = (r1 - r0 + 3) / 4, steps = tiles * batches;

  float4 a[SK_BLOCKS_F32][4];
  auto load = [&](int step) {
    const int row = r0 + (step / batches) * 4, kb = b0 + (step % batches) * SK_BLOCKS_F32;
#pragma unroll
    for (int i = 0; i < SK_BLOCKS_F32; ++i) {
      const int k = (kb + i) * 128 + lane * 4;
      const bool in = kb + i < b1 && k < K;
#pragma unroll
      for (int r = 0; r < 4; ++r)
        a[i][r] = in && row + r < r1 ? __ldcs(reinterpret_cast<const float4*>(w + (size_t)(row + r) * K + k))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  if (steps > 0) load(0);
  for (int i = tid; i < M * KB * 32; i += SK_THREADS) {
    const int m = i / (KB * 32), k = (i - m * KB * 32) * 4;
    reinterpret_cast<float4*>(xs)[i] = k < K ? __ldg(reinterpret_cast<const float4*>(x + (size_t)m * K + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  float2 acc[4][M];
  for (int step = 0; step < steps; ++step) {
    const int t = step / batches, bt = step - t * batches, kb = b0 + bt * SK_BLOCKS_F32;
    if (bt == 0)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int m = 0; m < M; ++m) acc[r][m] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < SK_BLOCKS_F32; ++i) {
      if (kb + i >= b1) break;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const float4 v = reinterpret_cast<const float4*>(xs)[(m * KB + kb + i) * 32 + lane];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          acc[r][m] = __ffma2_rn(make_float2(a[i][r].x, a[i][r].y), make_float2(v.x, v.y), acc[r][m]);
          acc[r][m] = __ffma2_rn(make_float2(a[i][r].z, a[i][r].w), make_float2(v.z, v.w), acc[r][m]);
        }
      }
    }
    if (step + 1 < steps) load(step + 1);
    if (bt + 1 == batches) {
      float v[4 * M];      // value m * 4 + r
#pragma unroll
      for (int m = 0; m < M; ++m)
#pragma unroll
        for (int r = 0; r < 4; ++r) v[m * 4 + r] = acc[r][m].x + acc[r][m].y;
      int base = 0;
      reduce_rec<4 * M, 16>(v, base, lane);
      constexpr int FC = final_cnt(4 * M, 16), DUP = dup_mask(4 * M, 16);
      float* mine = red + (t & 1) * SK_WARPS * 128;
      if ((lane & DUP) == 0) {
#pragma unroll
        for (int i = 0; i < FC; ++i) mine[warp * 128 + base + i] = v[i];
      }
      const int row0 = r0 + t * 4;
      sk_exchange(mine, group, KS, 4 * M, [&](int i, float s) {
        const int row = row0 + (i & 3), m = i >> 2;
        if (row < r1) y[(size_t)m * N + row] = s;
      });
    }
  }
}

}  // namespace spd
