// Several sequences through ONE pass over the weights (the batched, KV-heavy form of the verify
// step: the method's premise is that a target call is bound by streaming the parameters, Sec. 1 and
// Sec. 4 "Metrics", so B sequences should share that stream).  The rows of all sequences --
// B x (gamma + 1) for a verify step, B x 2 for a draft step -- go through each projection as one
// dense GEMM on the tcgen05 tensor cores (spd_gemm.cuh); attention, rotary embedding, cache
// append, the rejection rule and the commit stay per sequence: every sequence has its own cache,
// its own length and its own accepted count (Sec. 2.1's rule is stated per sequence).
#pragma once
#include "spd_kernel.cuh"
#include "spd_prefill.cuh"

namespace spd {

struct BatchSeq {
  DevState* st;
  int pos_base_t, pos_base_d;   // rows in front of the text in the target's / draft's cache
};

constexpr int BATCH_ROWS_MAX = 128;   // rows of a batched step: what its buffers are sized for

// Row (b, m) of a batched launch.  Verify: m = 0 the pending token, m >= 1 draft token m-1, cache row
// and rotary position origin_b + m.  Draft step j: the two rows [token before, token to extend] at
// origin_b + j - 1 + m (as in the single-sequence step).  Writes the embedding rows, each row's
// absolute cache row, and each sequence's origin.  An id outside [0, V) is read as 0 and reported.
__global__ void batch_embed_kernel(const BatchSeq* seqs, int B, int M, int draft, int j, const float* table, int d,
                                   int V, float* X, int* rowslot, int* origins, int* err) {
  pdl_wait();
  pdl_trigger();
  const int r = blockIdx.x, b = r / M, m = r - b * M;
  const DevState* st = seqs[b].st;
  const int origin = (draft ? seqs[b].pos_base_d : seqs[b].pos_base_t) + st->n_text;
  int id, slot;
  if (draft) {
    const int t = j - 1 + m;
    id = t < 0 ? st->prev : (t == 0 ? st->pending : st->d_ids[t - 1]);
    slot = origin + t;
  } else {
    id = m == 0 ? st->pending : st->d_ids[m - 1];
    slot = origin + m;
  }
  if ((unsigned)id >= (unsigned)V) {
    if (threadIdx.x == 0) atomicCAS(err, DEV_OK, DEV_BAD_TOKEN);
    id = 0;
  }
  if (threadIdx.x == 0) { rowslot[r] = slot; if (m == 0) origins[b] = origin; }
  const float4* src = reinterpret_cast<const float4*>(table + (size_t)id * d);
  float4* dst = reinterpret_cast<float4*>(X + (size_t)r * d);
  for (int i = threadIdx.x; i < (d >> 2); i += blockDim.x) dst[i] = src[i];
}

// qkv [slices][R][3d] (natural row order; K slices of the projection, added in slice order) -> rotary
// embedding on q and k at each row's own position; q goes to its sequence's query rows [M][d]
// (fp32), k and v are appended to its sequence's cache at the row's cache row.
__global__ void batch_rope_append_kernel(const float* qkv, int slices, int R, int M, int d, int dh, const int* rowslot,
                                         const float* cs, const float* sn, const ModelDev* mds, int layer) {
  pdl_wait();
  pdl_trigger();
  const int half = dh >> 1, quads = d >> 3, per_head = half >> 2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < R * quads; i += gridDim.x * blockDim.x) {
    const int r = i / quads, g = i - r * quads, h = g / per_head, j = (g - h * per_head) << 2, c0 = h * dh + j;
    const int b = r / M, m = r - b * M, pos = rowslot[r];
    const ModelDev& md = mds[b];
    const float4 c = *reinterpret_cast<const float4*>(cs + (size_t)pos * half + j);
    const float4 s = *reinterpret_cast<const float4*>(sn + (size_t)pos * half + j);
    const RopeQuad o = rope_quad(qkv, slices, (size_t)R * 3 * d, r, d, c0, half, c, s);
    float* q = md.qbuf + (size_t)m * d + c0;
    *reinterpret_cast<float4*>(q) = o.qa;
    *reinterpret_cast<float4*>(q + half) = o.qb;
    const size_t crow = (((size_t)layer * md.H + h) * md.max_seq + pos) * dh + j;   // cache: [L][H][max_seq][dh]
    __nv_bfloat16* kc = static_cast<__nv_bfloat16*>(md.kcache) + crow;
    __nv_bfloat16* vc = static_cast<__nv_bfloat16*>(md.vcache) + crow;
    *reinterpret_cast<uint2*>(kc) = pack4(o.ka);
    *reinterpret_cast<uint2*>(kc + half) = pack4(o.kb);
    *reinterpret_cast<uint2*>(vc) = pack4(o.va);
    *reinterpret_cast<uint2*>(vc + half) = pack4(o.vb);
  }
}

// Attention of every sequence's M rows over its own cache.  A work unit = (sequence, head, KV split)
// belongs to ONE WARP, which walks its rows in tiles of 8 KB (K and V) with a running softmax and
// synchronises with nobody: tiles arrive by cp.async into the warp's own three buffers.  Both products
// use mma.m16n8k16 with the M <= 8 query rows as rows 0..7 of the A operand and, since the rows 8..15
// would be padding, their bf16 lo parts there: one instruction does the hi and the lo product, and the two
// halves of the accumulator are added at the end.  The probabilities of a score tile are the A
// operand of the second product as they stand in the registers.  The splits of a head are merged by the
// warp that finishes last (no waiting); the result leaves as bf16 hi + lo [B * M][d].
//
// Bound by HBM (K/V bytes).  `splits` per head: as many units as warps fit on the device, so that all
// run at once and end together.  16 sequences, us a layer: 32 heads x 128, 1640 rows, M = 6: a CTA
// per unit with barriers between its score, softmax and output phases 122 -> this one 72;
// 12 heads x 64, 1030 rows, M = 2: 31 -> 16.5.
constexpr int BA_WARPS = 8, BA_STAGES = 3, BA_TILE_BYTES = 8192;   // a tile: K rows, then V rows
constexpr int BA_SMEM = BA_WARPS * BA_STAGES * BA_TILE_BYTES;

struct BatchAttnArgs {
  const ModelDev* mds;
  const int* origins;
  int B, H, d, M, layer, chain0, splits;
  float scale;
  float *part_o, *part_ml;      // [B * H * splits][8][dh], [..][8][2]
  unsigned* cnt;                // [B * H], zero between launches
  __nv_bfloat16 *o_hi, *o_lo;
};

// splits a sequence of `len` rows really uses: none shorter than two tiles
__device__ __forceinline__ int ba_splits(int splits, int len, int tile) {
  const int most = (len + 2 * tile - 1) / (2 * tile);
  return splits < most ? splits : most;
}

template <int DH>
__global__ void __launch_bounds__(BA_WARPS * 32, 1) batch_attn_kernel(const BatchAttnArgs a) {
  extern __shared__ __align__(1024) char ba_sm[];
  constexpr int ROWB = DH * 2, CPR = ROWB / 16, T = BA_TILE_BYTES / 2 / ROWB, ND = DH / 16;   // T = 16 or 32 positions
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gq = lane >> 2, tq = lane & 3, mat = lane >> 3, rr = lane & 7;
  char* buf = ba_sm + warp * BA_STAGES * BA_TILE_BYTES;
  // neighbouring units go to different SMs
  const int units = a.B * a.H * a.splits, stride = gridDim.x * BA_WARPS;
  for (int unit = warp * gridDim.x + blockIdx.x; unit < units; unit += stride) {
    const int sp = unit % a.splits, bh = unit / a.splits, h = bh % a.H, b = bh / a.H;
    const int origin = a.origins[b], len = origin + a.chain0 + a.M;
    const int ns = ba_splits(a.splits, len, T);
    if (sp >= ns) continue;
    const int Lc = ((len + ns - 1) / ns + T - 1) / T * T, p0 = min(len, sp * Lc), p1 = min(len, p0 + Lc);
    const ModelDev& md = a.mds[b];
    const size_t head = ((size_t)a.layer * a.H + h) * md.max_seq * ROWB;
    const char* Kg = static_cast<const char*>(md.kcache) + head;
    const char* Vg = static_cast<const char*>(md.vcache) + head;
    const int tiles = (p1 - p0 + T - 1) / T;
    auto request = [&](int t) {
      if (t < tiles) {
        char* Kt = buf + (t % BA_STAGES) * BA_TILE_BYTES;
        char* Vt = Kt + BA_TILE_BYTES / 2;
        const int c0 = p0 + t * T;
#pragma unroll
        for (int i = lane; i < T * CPR; i += 32) {
          const int r = i / CPR, c = i % CPR, dst = r * ROWB + ((c ^ (r & 7)) << 4);
          if (c0 + r < p1) {
            const size_t g = (size_t)(c0 + r) * ROWB + c * 16;
            cp_async16(Kt + dst, Kg + g);
            cp_async16(Vt + dst, Vg + g);
          } else {      // masked below, but must not hold NaN patterns
            *reinterpret_cast<uint4*>(Kt + dst) = make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4*>(Vt + dst) = make_uint4(0, 0, 0, 0);
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");   // (possibly empty: keeps the group count in step)
    };
    request(0);
    request(1);
    // query row gq: hi parts as A rows 0..7, lo parts as rows 8..15
    uint32_t qa[ND][4];
    const float* qr = md.qbuf + (size_t)gq * a.d + h * DH;
#pragma unroll
    for (int k = 0; k < ND; ++k)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 x = gq < a.M ? __ldcg(reinterpret_cast<const float2*>(qr + k * 16 + j * 8 + 2 * tq)) : make_float2(0.f, 0.f);
        qa[k][2 * j] = pack_bf16(x.x, x.y);
        qa[k][2 * j + 1] = pack_bf16(x.x - bf16lo(qa[k][2 * j]), x.y - bf16hi(qa[k][2 * j]));
      }
    float acc[DH / 8][4];
#pragma unroll
    for (int i = 0; i < DH / 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    float mx = -INFINITY, sum = 0.f;
    const int limit = origin + a.chain0 + gq;        // last position row gq attends
    for (int t = 0; t < tiles; ++t) {
      request(t + 2);
      asm volatile("cp.async.wait_group 2;" ::: "memory");
      __syncwarp();
      const uint32_t Kt = smem_u32(buf + (t % BA_STAGES) * BA_TILE_BYTES), Vt = Kt + BA_TILE_BYTES / 2;
      float s[T / 8][4];
#pragma unroll
      for (int i = 0; i < T / 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
#pragma unroll
      for (int k = 0; k < ND; ++k)
#pragma unroll
        for (int p = 0; p < T / 16; ++p) {
          const int r = p * 16 + (mat >> 1) * 8 + rr, c = (k * 2 + (mat & 1)) ^ (r & 7);
          uint32_t b0, b1, b2, b3;
          ldsm4(Kt + r * ROWB + c * 16, b0, b1, b2, b3);
          mma_bf16(s[2 * p], qa[k][0], qa[k][1], qa[k][2], qa[k][3], b0, b1);
          mma_bf16(s[2 * p + 1], qa[k][0], qa[k][1], qa[k][2], qa[k][3], b2, b3);
        }
      float sv[T / 8][2], nm = mx;
#pragma unroll
      for (int i = 0; i < T / 8; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          sv[i][j] = p0 + t * T + i * 8 + 2 * tq + j <= limit ? (s[i][j] + s[i][2 + j]) * a.scale : -INFINITY;
          nm = fmaxf(nm, sv[i][j]);
        }
      nm = fmaxf(nm, __shfl_xor_sync(0xffffffffu, nm, 1));
      nm = fmaxf(nm, __shfl_xor_sync(0xffffffffu, nm, 2));
      const float base = nm == -INFINITY ? 0.f : nm;      // nothing visible yet: every exp below is 0
      const float rescale = expf(mx - base);              // (first tile: exp(-inf) = 0)
      mx = nm;
      sum *= rescale;
#pragma unroll
      for (int i = 0; i < DH / 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] *= rescale;
#pragma unroll
      for (int p = 0; p < T / 16; ++p) {
        uint32_t pa[4];        // probabilities of 16 positions: hi rows, lo rows
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float e0 = expf(sv[2 * p + j][0] - base), e1 = expf(sv[2 * p + j][1] - base);
          sum += e0 + e1;
          pa[2 * j] = pack_bf16(e0, e1);
          pa[2 * j + 1] = pack_bf16(e0 - bf16lo(pa[2 * j]), e1 - bf16hi(pa[2 * j]));
        }
#pragma unroll
        for (int i = 0; i < ND; ++i) {
          const int r = p * 16 + (mat & 1) * 8 + rr, c = (i * 2 + (mat >> 1)) ^ (r & 7);
          uint32_t b0, b1, b2, b3;
          ldsm4_trans(Vt + r * ROWB + c * 16, b0, b1, b2, b3);
          mma_bf16(acc[2 * i], pa[0], pa[1], pa[2], pa[3], b0, b1);
          mma_bf16(acc[2 * i + 1], pa[0], pa[1], pa[2], pa[3], b2, b3);
        }
      }
      __syncwarp();      // the buffer is requested again in the next round
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    const size_t orow = ((size_t)b * a.M + gq) * a.d + h * DH;
    if (ns == 1) {
      if (gq < a.M) {
        const float inv = 1.0f / sum;
#pragma unroll
        for (int i = 0; i < DH / 8; ++i) {
          const float x0 = (acc[i][0] + acc[i][2]) * inv, x1 = (acc[i][1] + acc[i][3]) * inv;
          const uint32_t hw = pack_bf16(x0, x1);
          *reinterpret_cast<uint32_t*>(a.o_hi + orow + i * 8 + 2 * tq) = hw;
          *reinterpret_cast<uint32_t*>(a.o_lo + orow + i * 8 + 2 * tq) = pack_bf16(x0 - bf16lo(hw), x1 - bf16hi(hw));
        }
      }
      continue;
    }
    float* po = a.part_o + (size_t)bh * a.splits * 8 * DH;
    float* pml = a.part_ml + (size_t)bh * a.splits * 16;
    if (gq < a.M) {
#pragma unroll
      for (int i = 0; i < DH / 8; ++i)
        __stcg(reinterpret_cast<float2*>(po + ((size_t)sp * 8 + gq) * DH + i * 8 + 2 * tq),
               make_float2(acc[i][0] + acc[i][2], acc[i][1] + acc[i][3]));
      if (tq == 0) __stcg(reinterpret_cast<float2*>(pml + ((size_t)sp * 8 + gq) * 2), make_float2(mx, sum));
    }
    __threadfence();
    __syncwarp();
    unsigned old = 0;
    if (lane == 0) old = atomicAdd(a.cnt + bh, 1u);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old != (unsigned)ns - 1u) continue;
    __threadfence();
    if (gq < a.M) {
      float gm = -INFINITY, den = 0.f;
      for (int s2 = 0; s2 < ns; ++s2) gm = fmaxf(gm, __ldcg(pml + ((size_t)s2 * 8 + gq) * 2));
#pragma unroll
      for (int i = 0; i < DH / 8; ++i) acc[i][0] = acc[i][1] = 0.f;
      for (int s2 = 0; s2 < ns; ++s2) {
        const float2 ml = __ldcg(reinterpret_cast<const float2*>(pml + ((size_t)s2 * 8 + gq) * 2));
        const float w = ml.x == -INFINITY ? 0.f : expf(ml.x - gm);
        den = fmaf(w, ml.y, den);
#pragma unroll
        for (int i = 0; i < DH / 8; ++i) {
          const float2 o = __ldcg(reinterpret_cast<const float2*>(po + ((size_t)s2 * 8 + gq) * DH + i * 8 + 2 * tq));
          acc[i][0] = fmaf(w, o.x, acc[i][0]);
          acc[i][1] = fmaf(w, o.y, acc[i][1]);
        }
      }
      const float inv = 1.0f / den;
#pragma unroll
      for (int i = 0; i < DH / 8; ++i) {
        const float x0 = acc[i][0] * inv, x1 = acc[i][1] * inv;
        const uint32_t hw = pack_bf16(x0, x1);
        *reinterpret_cast<uint32_t*>(a.o_hi + orow + i * 8 + 2 * tq) = hw;
        *reinterpret_cast<uint32_t*>(a.o_lo + orow + i * 8 + 2 * tq) = pack_bf16(x0 - bf16lo(hw), x1 - bf16hi(hw));
      }
    }
    if (lane == 0) a.cnt[bh] = 0u;
  }
}

// ---- sampling.  CTAs of ROW_THREADS threads per row or sequence (a batch has enough of them to fill
// the device); the row is read from L2 a few times instead of being kept anywhere.

// max and sum of exp of logits / T over a row, each element one IEEE operation at a time (as the
// single-sequence path): every CTA of the row over its slice, then merged
struct RowStats { float mx, sum; };
struct StatScratch { float red[ROW_WARPS]; RowStats part[ROW_CTAS_MAX]; };
__device__ RowStats row_stats(const float* row, int V, float T, const RowSlice& rs, StatScratch* sc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int VC = (V + rs.C - 1) / rs.C, s0 = min(V, rs.rank * VC), s1 = min(V, s0 + VC);
  float mx = -INFINITY;
#pragma unroll 8
  for (int k = s0 + threadIdx.x; k < s1; k += ROW_THREADS) mx = fmaxf(mx, div_t(ldcg(row + k), T));
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) sc->red[warp] = mx;
  __syncthreads();
  mx = sc->red[lane];
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  __syncthreads();
  float sum = 0.f;
#pragma unroll 8
  for (int k = s0 + threadIdx.x; k < s1; k += ROW_THREADS) sum += expf(__fsub_rn(div_t(ldcg(row + k), T), mx));
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) sc->red[warp] = sum;
  __syncthreads();
  sum = sc->red[lane];
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (rs.C == 1) return RowStats{mx, sum};
  if (warp == 0 && lane < rs.C) { store_in_cta(&sc->part[rs.rank].mx, lane, mx); store_in_cta(&sc->part[rs.rank].sum, lane, sum); }
  cluster_sync_all_threads();
  RowStats r{-INFINITY, 0.f};
  for (int c = 0; c < rs.C; ++c) r.mx = fmaxf(r.mx, sc->part[c].mx);
  for (int c = 0; c < rs.C; ++c)
    if (sc->part[c].mx != -INFINITY) r.sum += sc->part[c].sum * expf(sc->part[c].mx - r.mx);
  return r;
}

// (max, sum exp) of every row -> stats [rows]; with probs also the probability rows (the truncated path
// needs them whole).  Row i reads logits row first + i * stride.
__global__ void __launch_bounds__(ROW_THREADS) batch_softmax_kernel(const float* logits, int first, int stride, int V,
                                                                    float temperature, RowStats* stats, float* probs) {
  __shared__ StatScratch sc;
  pdl_wait();
  pdl_trigger();
  const float* row = logits + ((size_t)first + (size_t)blockIdx.x * stride) * V;
  const RowStats rs = row_stats(row, V, temperature, RowSlice{0, 1}, &sc);
  if (threadIdx.x == 0) stats[blockIdx.x] = rs;
  if (probs) {
    float* out = probs + (size_t)blockIdx.x * V;
#pragma unroll 8
    for (int k = threadIdx.x; k < V; k += ROW_THREADS) out[k] = prob_of(ldcg(row + k), temperature, rs.mx, rs.sum);
  }
}

// Draft step j of every sequence (C CTAs each): x_j drawn from q_j = softmax(logits / T) of the sequence's
// second row (the token being extended), or its arg-max when greedy; q_j is kept as row j of the
// sequence's draft distributions [B][gamma][V].  probs: the truncated rows [B][V], or NULL.
__global__ void __launch_bounds__(ROW_THREADS) batch_draft_sample_kernel(const BatchSeq* seqs, int C,
                                                                         const float* logits, const float* probs, int V, int gamma, int j, int greedy,
                                                                         float temperature, const float* u, float* q_all, int* ids_out) {
  __shared__ RowScratch sc;
  __shared__ StatScratch ss;
  const RowSlice rs = row_slice(C);
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x / C;
  const float* lrow = logits + ((size_t)b * 2 + 1) * V;
  int tok;
  bool mine = rs.rank == 0;
  if (greedy) {
    rows_argmax([&](int, int k) { return ldcg(lrow + k); }, 1, V, rs, &sc);
    tok = sc.arg[0];
  } else {
    const float* prow = probs ? probs + (size_t)b * V : nullptr;
    const RowStats st = probs ? RowStats{0.f, 1.f} : row_stats(lrow, V, temperature, rs, &ss);
    auto wf = [&](int k) { return prow ? ldcg(prow + k) : prob_of(ldcg(lrow + k), temperature, st.mx, st.sum); };
    float* q = q_all + ((size_t)b * gamma + j) * V;
    const RowMass m = row_mass(wf, [&](int k, float w) { stcg(q + k, w); }, V, rs, &sc);
    mine = row_pick(wf, V, m, u[(size_t)b * gamma + j], rs, &sc, tok);
  }
  if (mine && threadIdx.x == 0) {
    seqs[b].st->d_ids[j] = tok;
    ids_out[b * gamma + j] = tok;      // all sequences' ids together for the caller
  }
}

// The rejection rule and the commit, C CTAs per sequence (Sec. 2.1): the target's rows are logits
// [B][gamma+1][V] with their statistics, or probability rows when truncated (greedy: only the arg-max of
// the logits is used); q_all [B][gamma][V] the draft's.  Each sequence advances by its own count.
__global__ void __launch_bounds__(ROW_THREADS) batch_verify_kernel(const BatchSeq* seqs, int C, const float* logits,
                                                                   const RowStats* stats, const float* probs, const float* q_all,
                                                                   const float* u, int gamma, int V, int greedy, float temperature,
                                                                   int* n_acc, int* next) {
  __shared__ RowScratch sc;
  __shared__ int s_ids[MAX_M];
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x / C;
  const RowSlice rs = row_slice(C);
  DevState* st = seqs[b].st;
  if (threadIdx.x < gamma) {
    const int x = st->d_ids[threadIdx.x];
    s_ids[threadIdx.x] = (unsigned)x < (unsigned)V ? x : 0;   // the embedding kernel has flagged it
  }
  __syncthreads();
  const size_t row0 = (size_t)b * (gamma + 1);
  auto pv = [&](int j, int k) {
    if (probs) return ldcg(probs + (row0 + j) * V + k);
    const float l = ldcg(logits + (row0 + j) * V + k);
    return greedy ? l : prob_of(l, temperature, stats[row0 + j].mx, stats[row0 + j].sum);
  };
  auto qv = [&](int j, int k) { return ldcg(q_all + ((size_t)b * gamma + j) * V + k); };
  int r, tok;
  const bool mine = rule_rows(pv, qv, s_ids, u ? u + row0 : nullptr, gamma, V, greedy, rs, &sc, gridDim.x / C, r, tok);
  if (mine && threadIdx.x == 0) {
    st->n_acc = r;
    st->next = tok;
    st->n_text += r + 1;
    st->prev = r >= 1 ? s_ids[r - 1] : st->pending;
    st->pending = tok;
    st->block += 1;
    if (n_acc) n_acc[b] = r;
    if (next) next[b] = tok;
  }
}

}  // namespace spd
