// Elementwise kernels around the dense linear maps of the prefill, the batched steps and the image
// adapter: bf16 hi/lo split, residual + RMSNorm, rotary embedding + cache append.  All are bound by
// memory or by launch latency: 16-byte loads, 8-byte bf16 stores, dependent launches.
#pragma once
#include "spd_device.cuh"

namespace spd {

// ------------------------------------------------------------------------------ elementwise

__device__ __forceinline__ uint32_t split_pair(float a, float b, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
  lo = *reinterpret_cast<const uint32_t*>(&l);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// four fp32 values -> bf16 hi + lo at element offset o (a multiple of 4)
__device__ __forceinline__ void store_split4(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t o, float4 x) {
  uint2 h, l;
  h.x = split_pair(x.x, x.y, l.x);
  h.y = split_pair(x.z, x.w, l.y);
  *reinterpret_cast<uint2*>(hi + o) = h;
  *reinterpret_cast<uint2*>(lo + o) = l;
}
__device__ __forceinline__ uint2 pack4(float4 x) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// fp32 [R][K] -> hi/lo bf16 [R][K]; n is a multiple of 8 (K is), the rows 16-byte aligned or not at all
__global__ void split_rows_kernel(const float* x, __nv_bfloat16* hi, __nv_bfloat16* lo, size_t n, int aligned) {
  pdl_wait();
  pdl_trigger();
  for (size_t i = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) * 4; i < n; i += (size_t)gridDim.x * blockDim.x * 4) {
    const float4 v = aligned ? *reinterpret_cast<const float4*>(x + i) : make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
    store_split4(hi, lo, i, v);
  }
}

// x[row] += sum over the K slices of a projection's partial products (in slice order), then the
// RMSNorm of the updated row with `gain`, split into hi/lo bf16.  slices = 0: only the norm.
__global__ void __launch_bounds__(256) resid_rms_split_kernel(float* x, const float* part, int slices, size_t slice_stride,
                                                              const float* gain, float eps, int d, __nv_bfloat16* hi,
                                                              __nv_bfloat16* lo) {
  __shared__ float red[8];
  constexpr int PER = 4096 / 4 / 256;     // float4 per thread: rows of up to 4096 columns stay in registers
  float* row = x + (size_t)blockIdx.x * d;
  const float* prow = part + (size_t)blockIdx.x * d;
  const int d4 = d >> 2;
  float4 v[PER], g[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) {         // gains are weights: they need no predecessor
    const int k4 = threadIdx.x + i * 256;
    if (k4 < d4) g[i] = __ldg(reinterpret_cast<const float4*>(gain) + k4);
  }
  pdl_wait();
  pdl_trigger();
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int k4 = threadIdx.x + i * 256;
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k4 < d4) {
      v[i] = reinterpret_cast<const float4*>(row)[k4];
      float4 p[8];   // all slices of this piece travel together, then they are added in slice order
#pragma unroll
      for (int s = 0; s < 8; ++s)
        if (s < slices) p[s] = reinterpret_cast<const float4*>(prow + (size_t)s * slice_stride)[k4];
#pragma unroll
      for (int s = 0; s < 8; ++s)
        if (s < slices) { v[i].x += p[s].x; v[i].y += p[s].y; v[i].z += p[s].z; v[i].w += p[s].w; }
      if (slices > 0) reinterpret_cast<float4*>(row)[k4] = v[i];
      ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += red[w];
  const float inv = 1.0f / sqrtf(tot / (float)d + eps);
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int k4 = threadIdx.x + i * 256;
    if (k4 < d4)
      store_split4(hi, lo, (size_t)blockIdx.x * d + (size_t)k4 * 4,
                   make_float4((v[i].x * inv) * g[i].x, (v[i].y * inv) * g[i].y, (v[i].z * inv) * g[i].z, (v[i].w * inv) * g[i].w));
  }
}

// Four neighbouring rotary pairs of one head of one row: columns c0 .. c0+3 and c0 + dh/2 .. of q, k and v,
// each the sum of `slices` partial products [slices][R][3d] in slice order.
struct RopeQuad {
  float4 qa, qb, ka, kb, va, vb;
};
__device__ __forceinline__ float4 sum_slices(const float* p, int slices, size_t stride) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s = 0; s < slices; ++s) {
    const float4 x = *reinterpret_cast<const float4*>(p + (size_t)s * stride);
    v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
  }
  return v;
}
__device__ __forceinline__ RopeQuad rope_quad(const float* qkv, int slices, size_t stride, int r, int d, int c0, int half,
                                              float4 c, float4 s) {
  const float* row = qkv + (size_t)r * 3 * d + c0;
  RopeQuad o;
  const float4 qa = sum_slices(row, slices, stride), qb = sum_slices(row + half, slices, stride);
  const float4 ka = sum_slices(row + d, slices, stride), kb = sum_slices(row + d + half, slices, stride);
  o.va = sum_slices(row + 2 * d, slices, stride);
  o.vb = sum_slices(row + 2 * d + half, slices, stride);
  o.qa = make_float4(qa.x * c.x - qb.x * s.x, qa.y * c.y - qb.y * s.y, qa.z * c.z - qb.z * s.z, qa.w * c.w - qb.w * s.w);
  o.qb = make_float4(qb.x * c.x + qa.x * s.x, qb.y * c.y + qa.y * s.y, qb.z * c.z + qa.z * s.z, qb.w * c.w + qa.w * s.w);
  o.ka = make_float4(ka.x * c.x - kb.x * s.x, ka.y * c.y - kb.y * s.y, ka.z * c.z - kb.z * s.z, ka.w * c.w - kb.w * s.w);
  o.kb = make_float4(kb.x * c.x + ka.x * s.x, kb.y * c.y + ka.y * s.y, kb.z * c.z + ka.z * s.z, kb.w * c.w + ka.w * s.w);
  return o;
}

// qkv [slices][R][3d] (natural row order) of prompt rows at positions 0.. -> rotary on q and k (pairs
// (i, i + dh/2)), q split into hi/lo [R][d], k and v appended to the cache of one layer [H][max_seq][dh].
__global__ void rope_kv_kernel(const float* qkv, int slices, int R, int d, int dh, const float* cs, const float* sn,
                               __nv_bfloat16* q_hi, __nv_bfloat16* q_lo, __nv_bfloat16* kc, __nv_bfloat16* vc, int max_seq) {
  pdl_wait();
  pdl_trigger();
  const int half = dh >> 1, quads = d >> 3, per_head = half >> 2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < R * quads; i += gridDim.x * blockDim.x) {
    const int r = i / quads, g = i - r * quads, h = g / per_head, j = (g - h * per_head) << 2, c0 = h * dh + j;
    const float4 c = *reinterpret_cast<const float4*>(cs + (size_t)r * half + j);
    const float4 s = *reinterpret_cast<const float4*>(sn + (size_t)r * half + j);
    const RopeQuad o = rope_quad(qkv, slices, (size_t)R * 3 * d, r, d, c0, half, c, s);
    store_split4(q_hi, q_lo, (size_t)r * d + c0, o.qa);
    store_split4(q_hi, q_lo, (size_t)r * d + c0 + half, o.qb);
    const size_t crow = ((size_t)h * max_seq + r) * dh + j;
    *reinterpret_cast<uint2*>(kc + crow) = pack4(o.ka);
    *reinterpret_cast<uint2*>(kc + crow + half) = pack4(o.kb);
    *reinterpret_cast<uint2*>(vc + crow) = pack4(o.va);
    *reinterpret_cast<uint2*>(vc + crow + half) = pack4(o.vb);
  }
}

}  // namespace spd
