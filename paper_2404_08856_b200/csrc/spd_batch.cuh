// Several sequences through ONE pass over the weights (the batched, KV-heavy form of the verify
// step: the method's premise is that a target call is bound by streaming the parameters, Sec. 1 and
// Sec. 4 "Metrics", so B sequences should share that stream).  The rows of all sequences --
// B x (gamma + 1) for a verify step, B x 2 for a draft step -- go through each projection as one
// dense GEMM on the tcgen05 tensor cores (spd_prefill.cuh); attention, rotary embedding, cache
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

constexpr int BATCH_ROWS_MAX = 128;   // one 128-row tile of the tensor-core GEMM

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

// Attention of every sequence's M rows over its own cache.  Work unit = (sequence, head, KV split),
// the single-sequence unit of attn_phase_mma (partial results of a head merged by the CTA that
// finishes its last split); the units of ALL sequences form one list that a grid of persistent CTAs
// walks with stride gridDim.x, so a CTA's next unit usually belongs to another sequence and no CTA
// waits for another.  `chain0`: block-row offset of row 0 (verify: 0; draft step j: j - 1); row m
// attends the rows from the origin up to its own.
// `max_split`: KV splits per head at most -- with B sequences there are enough (sequence, head) pairs
// to fill the grid, so heads are cut no further than needed (fewer partial results to merge).
// o_hi / o_lo: every sequence's output rows as one matrix [B * M][d] split into bf16 hi + lo (the
// operand of the output projection).
template <int M>
__global__ void __launch_bounds__(CONSUMER_THREADS, 2) batch_attn_kernel(const ModelDev* mds, const int* origins, int B,
                                                                      int layer, int chain0, int xbytes, int max_split,
                                                                      __nv_bfloat16* o_hi, __nv_bfloat16* o_lo) {
  extern __shared__ __align__(1024) char bsm[];
  pdl_wait();
  pdl_trigger();
  Ctrl* ctl = reinterpret_cast<Ctrl*>(bsm);
  char* xs = bsm + CTRL_BYTES;
  if (threadIdx.x < M) {
    const int top = chain0 + (int)threadIdx.x;          // highest block row this row attends (-1: none)
    ctl->sees[threadIdx.x] = top < 0 ? 0u : ((2u << top) - 1u);
  }
  __syncthreads();
  const int umax = mds[0].H * max_split;                // most units a sequence can have
  for (int g = blockIdx.x; g < B * umax; g += gridDim.x) {
    const int b = g / umax, u = g - b * umax;
    ModelDev md = mds[b];
    md.nsplit = max_split;
    const int units = md.H * eff_nsplit(md, origins[b] + chain0 + M);
    if (u >= units) continue;
    // one unit: the phase's own loop runs once for "CTA u of a grid of `units`"
    const size_t row0 = (size_t)b * M * md.d;
    attn_phase_mma<M, true>(md, layer, origins[b], chain0 + M, u, units, xs, xbytes, ctl, o_hi + row0, o_lo + row0);
    named_sync(1, CONSUMER_THREADS);
  }
}

// ---- sampling.  CTAs of ROW_THREADS threads per row or sequence (a batch has enough of them to fill
// the device); the row is read from L2 a few times instead of being kept anywhere.

// max and sum of exp of logits / T over a row, each step one IEEE operation (as the single-sequence path)
struct RowStats { float mx, sum; };
__device__ RowStats row_stats(const float* row, int V, float T, float* red /*[ROW_WARPS]*/) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float mx = -INFINITY;
#pragma unroll 8
  for (int k = threadIdx.x; k < V; k += ROW_THREADS) mx = fmaxf(mx, __fdiv_rn(ldcg(row + k), T));
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) red[warp] = mx;
  __syncthreads();
  mx = red[lane];
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  __syncthreads();
  float sum = 0.f;
#pragma unroll 8
  for (int k = threadIdx.x; k < V; k += ROW_THREADS) sum += expf(__fsub_rn(__fdiv_rn(ldcg(row + k), T), mx));
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) red[warp] = sum;
  __syncthreads();
  sum = red[lane];
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return RowStats{mx, sum};
}

// (max, sum exp) of every row -> stats [rows]; with probs also the probability rows (the truncated path
// needs them whole).  Row i reads logits row first + i * stride.
__global__ void __launch_bounds__(ROW_THREADS) batch_softmax_kernel(const float* logits, int first, int stride, int V,
                                                                    float temperature, RowStats* stats, float* probs) {
  __shared__ float red[ROW_WARPS];
  pdl_wait();
  pdl_trigger();
  const float* row = logits + ((size_t)first + (size_t)blockIdx.x * stride) * V;
  const RowStats rs = row_stats(row, V, temperature, red);
  if (threadIdx.x == 0) stats[blockIdx.x] = rs;
  if (probs) {
    float* out = probs + (size_t)blockIdx.x * V;
#pragma unroll 8
    for (int k = threadIdx.x; k < V; k += ROW_THREADS) out[k] = prob_of(ldcg(row + k), temperature, rs.mx, rs.sum);
  }
}

// Draft step j of every sequence (one CTA each): x_j drawn from q_j = softmax(logits / T) of the sequence's
// second row (the token being extended), or its arg-max when greedy; q_j is kept as row j of the
// sequence's draft distributions [B][gamma][V].  probs: the truncated rows [B][V], or NULL.
__global__ void __launch_bounds__(ROW_THREADS) batch_draft_sample_kernel(const BatchSeq* seqs, const float* logits,
                                                                         const float* probs, int V, int gamma, int j, int greedy,
                                                                         float temperature, const float* u, float* q_all) {
  __shared__ RowScratch sc;
  __shared__ float red[ROW_WARPS];
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x;
  const RowSlice rs{0, 1};
  const float* lrow = logits + ((size_t)b * 2 + 1) * V;
  int tok;
  if (greedy) {
    rows_argmax([&](int, int k) { return ldcg(lrow + k); }, 1, V, rs, &sc);
    tok = sc.arg[0];
  } else {
    const float* prow = probs ? probs + (size_t)b * V : nullptr;
    const RowStats st = probs ? RowStats{0.f, 1.f} : row_stats(lrow, V, temperature, red);
    auto wf = [&](int k) { return prow ? ldcg(prow + k) : prob_of(ldcg(lrow + k), temperature, st.mx, st.sum); };
    float* q = q_all + ((size_t)b * gamma + j) * V;
    const unsigned long long Z = row_mass(wf, [&](int k, float w) { stcg(q + k, w); }, V, rs, &sc);
    row_pick(wf, V, Z, u[(size_t)b * gamma + j], rs, &sc, tok);
  }
  if (threadIdx.x == 0) seqs[b].st->d_ids[j] = tok;
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
  const bool mine = rule_rows(pv, qv, s_ids, u ? u + row0 : nullptr, gamma, V, greedy, rs, &sc, r, tok);
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
