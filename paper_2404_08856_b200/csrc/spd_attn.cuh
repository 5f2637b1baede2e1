// Causal attention of the prefill (Eq. 1's decoder over all prompt rows at once): one CTA of four warps
// takes 64 query rows of one head and walks the cached K/V rows in tiles of 64 with a running
// softmax, so scores and probabilities never leave the registers.
//
// Both products run on the tensor cores with K and V as they are cached (bf16); the query rows and the
// probabilities are fp32 quantities fed as bf16 hi + lo.  Scores, softmax and the output accumulate in
// fp32.  K/V tiles are double-buffered with cp.async, 16-byte pieces swizzled by row for ldmatrix.
// The query tiles with the longest rows are launched first, so the short ones fill the tail.
//
// What bounds it: MMA issue (two products, each twice for hi and lo: 4 x R^2 / 2 x d_head x 2 flops per
// head).  640 rows, 32 heads x 128: three launches through fp32 scores in HBM took 36 + 54 + 24 us a
// layer, this one 39.
#pragma once
#include "spd_engine.cuh"

namespace spd {

constexpr int PA_ROWS = 64, PA_KV = 64, PA_THREADS = 128;
__host__ __device__ constexpr int pa_smem(int dh) { return 2 * 2 * PA_KV * dh * 2; }

template <int DH>
__global__ void __launch_bounds__(PA_THREADS, 2)
prefill_attn_kernel(const __nv_bfloat16* q_hi, const __nv_bfloat16* q_lo, const __nv_bfloat16* kc, const __nv_bfloat16* vc,
                    int R, int H, int max_seq, float scale, __nv_bfloat16* o_hi, __nv_bfloat16* o_lo) {
  extern __shared__ __align__(1024) char pa_sm[];
  constexpr int ROWB = DH * 2, CPR = ROWB / 16, TILE = PA_KV * ROWB, ND = DH / 16;
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gq = lane >> 2, tq = lane & 3, mat = lane >> 3, rr = lane & 7;
  const int nq = (R + PA_ROWS - 1) / PA_ROWS;
  const int h = blockIdx.x % H, q0 = (nq - 1 - (int)(blockIdx.x / H)) * PA_ROWS;
  const int d = H * DH;
  const char* Kg = reinterpret_cast<const char*>(kc + (size_t)h * max_seq * DH);
  const char* Vg = reinterpret_cast<const char*>(vc + (size_t)h * max_seq * DH);
  const int kv_end = min(R, q0 + PA_ROWS);
  const int tiles = (kv_end + PA_KV - 1) / PA_KV;

  auto request = [&](int t) {
    char* Kt = pa_sm + (t & 1) * 2 * TILE;
    char* Vt = Kt + TILE;
    for (int i = tid; i < PA_KV * CPR; i += PA_THREADS) {
      const int r = i / CPR, c = i % CPR, dst = r * ROWB + ((c ^ (r & 7)) << 4);
      const int row = t * PA_KV + r;
      if (row < R) {
        cp_async16(Kt + dst, Kg + (size_t)row * ROWB + c * 16);
        cp_async16(Vt + dst, Vg + (size_t)row * ROWB + c * 16);
      } else {      // masked below, but must not hold NaN patterns
        *reinterpret_cast<uint4*>(Kt + dst) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(Vt + dst) = make_uint4(0, 0, 0, 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  request(0);

  // this warp's 16 query rows as A fragments, hi and lo
  const int ra = q0 + warp * 16 + gq, rb = ra + 8;
  uint32_t qh[ND][4], ql[ND][4];
#pragma unroll
  for (int k = 0; k < ND; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int row = (j & 1) ? rb : ra;
      const size_t o = (size_t)row * d + h * DH + k * 16 + (j >> 1) * 8 + 2 * tq;
      qh[k][j] = row < R ? *reinterpret_cast<const uint32_t*>(q_hi + o) : 0u;
      ql[k][j] = row < R ? *reinterpret_cast<const uint32_t*>(q_lo + o) : 0u;
    }
  float acc[DH / 8][4];
#pragma unroll
  for (int i = 0; i < DH / 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float mx[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};

  for (int t = 0; t < tiles; ++t) {
    if (t + 1 < tiles) {
      request(t + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const uint32_t Kt = smem_u32(pa_sm + (t & 1) * 2 * TILE), Vt = Kt + TILE;
    float s[PA_KV / 8][4];
#pragma unroll
    for (int i = 0; i < PA_KV / 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
#pragma unroll
    for (int k = 0; k < ND; ++k)
#pragma unroll
      for (int p = 0; p < PA_KV / 16; ++p) {
        const int r = p * 16 + (mat >> 1) * 8 + rr, c = (k * 2 + (mat & 1)) ^ (r & 7);
        uint32_t b0, b1, b2, b3;
        ldsm4(Kt + r * ROWB + c * 16, b0, b1, b2, b3);
        mma_bf16(s[2 * p], qh[k][0], qh[k][1], qh[k][2], qh[k][3], b0, b1);
        mma_bf16(s[2 * p + 1], qh[k][0], qh[k][1], qh[k][2], qh[k][3], b2, b3);
        mma_bf16(s[2 * p], ql[k][0], ql[k][1], ql[k][2], ql[k][3], b0, b1);
        mma_bf16(s[2 * p + 1], ql[k][0], ql[k][1], ql[k][2], ql[k][3], b2, b3);
      }
    // scale, causal mask (only the tiles that reach the diagonal need one), running maximum
    const bool diag = (t + 1) * PA_KV > q0 + warp * 16;
    float nm[2] = {mx[0], mx[1]};
#pragma unroll
    for (int i = 0; i < PA_KV / 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[i][j] *= scale;
        if (diag && t * PA_KV + i * 8 + 2 * tq + (j & 1) > ((j >> 1) ? rb : ra)) s[i][j] = -INFINITY;
        nm[j >> 1] = fmaxf(nm[j >> 1], s[i][j]);
      }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      nm[r] = fmaxf(nm[r], __shfl_xor_sync(0xffffffffu, nm[r], 1));
      nm[r] = fmaxf(nm[r], __shfl_xor_sync(0xffffffffu, nm[r], 2));
      const float rescale = mx[r] == -INFINITY ? 0.f : expf(mx[r] - nm[r]);
      mx[r] = nm[r];
      sum[r] *= rescale;
#pragma unroll
      for (int i = 0; i < DH / 8; ++i) { acc[i][2 * r] *= rescale; acc[i][2 * r + 1] *= rescale; }
    }
#pragma unroll
    for (int p = 0; p < PA_KV / 16; ++p) {
      uint32_t ph[4], pl[4];     // the probabilities of 16 positions as an A fragment, hi and lo
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = 2 * p + (j >> 1), o = (j & 1) * 2, r = j & 1;
        // (row 0 of the sequence sees position 0, so nm is finite once tile 0 has been seen)
        const float e0 = expf(s[i][o] - nm[r]), e1 = expf(s[i][o + 1] - nm[r]);
        sum[r] += e0 + e1;
        ph[j] = pack_bf16(e0, e1);
        pl[j] = pack_bf16(e0 - bf16lo(ph[j]), e1 - bf16hi(ph[j]));
      }
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        const int r = p * 16 + (mat & 1) * 8 + rr, c = (i * 2 + (mat >> 1)) ^ (r & 7);
        uint32_t b0, b1, b2, b3;
        ldsm4_trans(Vt + r * ROWB + c * 16, b0, b1, b2, b3);
        mma_bf16(acc[2 * i], ph[0], ph[1], ph[2], ph[3], b0, b1);
        mma_bf16(acc[2 * i + 1], ph[0], ph[1], ph[2], ph[3], b2, b3);
        mma_bf16(acc[2 * i], pl[0], pl[1], pl[2], pl[3], b0, b1);
        mma_bf16(acc[2 * i + 1], pl[0], pl[1], pl[2], pl[3], b2, b3);
      }
    }
    __syncthreads();     // the tile's buffer is requested again in the next round
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    sum[r] += __shfl_xor_sync(0xffffffffu, sum[r], 1);
    sum[r] += __shfl_xor_sync(0xffffffffu, sum[r], 2);
    const int row = r ? rb : ra;
    if (row >= R) continue;
    const float inv = 1.0f / sum[r];
#pragma unroll
    for (int i = 0; i < DH / 8; ++i) {
      const float x0 = acc[i][2 * r] * inv, x1 = acc[i][2 * r + 1] * inv;
      const uint32_t hw = pack_bf16(x0, x1), lw = pack_bf16(x0 - bf16lo(hw), x1 - bf16hi(hw));
      const size_t o = (size_t)row * d + h * DH + i * 8 + 2 * tq;
      *reinterpret_cast<uint32_t*>(o_hi + o) = hw;
      *reinterpret_cast<uint32_t*>(o_lo + o) = lw;
    }
  }
}

}  // namespace spd
