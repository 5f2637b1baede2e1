// Sampling primitives: integer inverse CDF, accept test, arg-max, the rejection rule.
//
// Drawing from a weight vector w with a uniform u is an inverse-CDF lookup in integers:
// W_k = trunc(w_k * 2^32), Z = sum W_k, t = floor(Z * floor(u * 2^24) / 2^24), result =
// the smallest k whose inclusive prefix sum exceeds t; Z == 0 falls back to argmax(w)
// (lowest index).  Integer sums make the result independent of the reduction tree.
// The acceptance rule and the residual follow Sec. 2.1 of the paper (p = target,
// q = draft): accept iff u < min(1, p/q); replacement ~ max(0, p - q) / sum.
#pragma once
#include "spd_device.cuh"

namespace spd {

__device__ __forceinline__ unsigned long long to_fixed(float w) {
  return static_cast<unsigned long long>(__fmul_rn(w, 4294967296.0f));  // cvt.rzi, exact scale
}

__device__ __forceinline__ unsigned long long threshold(unsigned long long Z, float u) {
  const unsigned long long u24 = static_cast<unsigned long long>(__fmul_rn(u, 16777216.0f));
  const unsigned long long lo = Z * u24, hi = __umul64hi(Z, u24);
  return (hi << 40) | (lo >> 24);
}

// min(1, p/q) with one IEEE division; q == 0 accepts iff p > 0.
__device__ __forceinline__ bool accept_test(float u, float p, float q) {
  float a;
  if (q == 0.0f) a = p > 0.0f ? 1.0f : 0.0f;
  else a = fminf(1.0f, __fdiv_rn(p, q));
  return u < a;
}

// ---- rows spread over a thread-block cluster
// The sampling kernels give a vocabulary row to a cluster of C CTAs of up to ROW_THREADS threads (C = 1 is
// an ordinary CTA; any whole number of warps works): CTA `rank` owns the contiguous slice [rank * VC, (rank + 1) * VC), a warp a contiguous
// piece of it, and the CTAs exchange their integer totals through each other's shared memory, one
// cluster barrier per draw.  One CTA of 256 threads needs 22 us for a draw from 32000 weights (its
// latency: every pass is 125 dependent loads deep), the grid-wide form in two launches 8 + 7 us.
constexpr int ROW_THREADS = 1024, ROW_WARPS = ROW_THREADS / 32, ROW_CTAS_MAX = 8;
__device__ __forceinline__ int row_warps() { return (int)(blockDim.x >> 5); }
constexpr int ARG_ROWS = 8;     // rows whose arg-max is taken together

struct RowScratch {
  unsigned long long wsum[ROW_WARPS];
  float wmax[ROW_WARPS];
  int widx[ROW_WARPS];
  unsigned long long tot[ROW_CTAS_MAX];            // every CTA's mass
  float cmax[ROW_CTAS_MAX];                        // its largest weight
  int cidx[ROW_CTAS_MAX];
  float amax[ARG_ROWS][ROW_WARPS];                 // arg-max of several rows at once
  int aidx[ARG_ROWS][ROW_WARPS];
  float gmax[ARG_ROWS][ROW_CTAS_MAX];
  int gidx[ARG_ROWS][ROW_CTAS_MAX];
  int arg[ARG_ROWS];
  int result;
  int first_reject;
};

struct RowSlice {
  int rank, C;      // this CTA among the C CTAs of its row
};
// Every CTA of the cluster has to be running before another one writes into its shared memory.
__device__ __forceinline__ RowSlice row_slice(int C) {
  if (C > 1) cluster_sync_all_threads();
  return RowSlice{(int)(blockIdx.x % C), C};
}

template <class T>
__device__ __forceinline__ void store_in_cta(T* p, int cta, T v) {   // p: this CTA's address of the word
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "");
  const uint32_t a = cluster_map(smem_u32(p), (unsigned)cta);
  if constexpr (sizeof(T) == 8)
    asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(*reinterpret_cast<unsigned long long*>(&v)) : "memory");
  else
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(*reinterpret_cast<unsigned*>(&v)) : "memory");
}

// the pieces of a slice: warp w of the CTA takes [k0, k1)
__device__ __forceinline__ void row_piece(const RowSlice& rs, int V, int warp, int& k0, int& k1) {
  const int VC = (V + rs.C - 1) / rs.C, s0 = min(V, rs.rank * VC), s1 = min(V, s0 + VC);
  const int nw = row_warps(), VW = (((s1 - s0 + nw - 1) / nw) + 31) & ~31;
  k0 = min(s1, s0 + warp * VW);
  k1 = min(s1, k0 + VW);
}

constexpr int ROW_UNROLL = 8;    // loads in flight per thread

// Masses of the row's weights; emit(k, w) sees every weight of this CTA's slice once.  Returns the row's
// total mass (the same in every CTA); the weights can then be drawn from with row_pick.
template <class WF, class EM>
__device__ unsigned long long row_mass(WF wf, EM emit, int V, const RowSlice& rs, RowScratch* sc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int k0, k1;
  row_piece(rs, V, warp, k0, k1);
  unsigned long long s = 0;
  float bm = -1.0f;
  int bi = 0x7fffffff;
  for (int kb = k0; kb < k1; kb += 32 * ROW_UNROLL) {
    float w[ROW_UNROLL];
#pragma unroll
    for (int i = 0; i < ROW_UNROLL; ++i) {
      const int k = kb + i * 32 + lane;
      w[i] = k < k1 ? wf(k) : -1.0f;
    }
#pragma unroll
    for (int i = 0; i < ROW_UNROLL; ++i) {
      const int k = kb + i * 32 + lane;
      if (k < k1) {
        s += to_fixed(w[i]);
        if (w[i] > bm) { bm = w[i]; bi = k; }
        emit(k, w[i]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    const float om = __shfl_xor_sync(0xffffffffu, bm, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (om > bm || (om == bm && oi < bi)) { bm = om; bi = oi; }
  }
  if (lane == 0) { sc->wsum[warp] = s; sc->wmax[warp] = bm; sc->widx[warp] = bi; }
  __syncthreads();
  if (warp == 0) {
    const bool on = lane < row_warps();
    s = on ? sc->wsum[lane] : 0ull; bm = on ? sc->wmax[lane] : -1.0f; bi = on ? sc->widx[lane] : 0x7fffffff;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      const float om = __shfl_xor_sync(0xffffffffu, bm, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (om > bm || (om == bm && oi < bi)) { bm = om; bi = oi; }
    }
    if (lane < rs.C) {
      store_in_cta(&sc->tot[rs.rank], lane, s);
      store_in_cta(&sc->cmax[rs.rank], lane, bm);
      store_in_cta(&sc->cidx[rs.rank], lane, bi);
    }
  }
  cluster_sync_all_threads();
  unsigned long long Z = 0;
  for (int c = 0; c < rs.C; ++c) Z += sc->tot[c];
  return Z;
}

// The token that uniform u draws from the weights of the preceding row_mass.  Exactly one CTA of the
// cluster, the one whose slice holds the token, returns true.
template <class WF>
__device__ bool row_pick(WF wf, int V, unsigned long long Z, float u, const RowSlice& rs, RowScratch* sc, int& tok) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (Z == 0) {      // no mass at all: the largest weight, lowest index on ties
    float m = sc->cmax[0];
    tok = sc->cidx[0];
    for (int c = 1; c < rs.C; ++c)
      if (sc->cmax[c] > m) { m = sc->cmax[c]; tok = sc->cidx[c]; }
    if (tok >= V) tok = 0;      // a row of NaN has no largest weight
    return rs.rank == 0;
  }
  const unsigned long long T = threshold(Z, u);
  unsigned long long base = 0;
  int cc = 0;
  while (cc < rs.C - 1 && T >= base + sc->tot[cc]) base += sc->tot[cc++];
  if (cc != rs.rank) return false;
  // the warp whose piece the running total crosses T in
  const unsigned long long own = lane < row_warps() ? sc->wsum[lane] : 0ull;
  unsigned long long inc = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  const unsigned over = __ballot_sync(0xffffffffu, T < base + inc);
  const int ww = over ? __ffs(over) - 1 : row_warps() - 1;
  base += __shfl_sync(0xffffffffu, inc - own, ww);
  if (warp == ww) {
    int k0, k1;
    row_piece(rs, V, warp, k0, k1);
    int found = max(k1 - 1, 0);
    constexpr int B = 16;          // 32-wide steps looked at together
    bool hit = false;
    for (int kb = k0; kb < k1 && !hit; kb += 32 * B) {
      unsigned long long m[B];
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const int k = kb + i * 32 + lane;
        m[i] = k < k1 ? to_fixed(wf(k)) : 0ull;
      }
#pragma unroll
      for (int i = 0; i < B; ++i) {
        if (hit) continue;
        // the step's total: three 32-bit sums of 27-bit parts
        const unsigned long long tot = (unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)(m[i] & 0x7ffffffull)) +
                                       ((unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)((m[i] >> 27) & 0x7ffffffull)) << 27) +
                                       ((unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)(m[i] >> 54)) << 54);
        if (T < base + tot) {
          unsigned long long pre = m[i];
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xffffffffu, pre, o);
            if (lane >= o) pre += t;
          }
          const unsigned mask = __ballot_sync(0xffffffffu, base + pre > T);
          found = kb + i * 32 + __ffs(mask) - 1;
          hit = true;
        } else {
          base += tot;
        }
      }
    }
    if (lane == 0) sc->result = found;
  }
  __syncthreads();
  tok = sc->result;
  __syncthreads();
  return true;
}

// One draw.
template <class WF>
__device__ bool row_sample(WF wf, int V, float u, const RowSlice& rs, RowScratch* sc, int& tok) {
  const unsigned long long Z = row_mass(wf, [](int, float) {}, V, rs, sc);
  return row_pick(wf, V, Z, u, rs, sc, tok);
}

// Arg-max (lowest index on ties) of n <= ARG_ROWS rows at once: f(j, k) = value k of row j; the results are
// left in sc->arg of every CTA.
template <class F>
__device__ void rows_argmax(F f, int n, int V, const RowSlice& rs, RowScratch* sc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int VC = (V + rs.C - 1) / rs.C, s0 = min(V, rs.rank * VC), s1 = min(V, s0 + VC);
  for (int j = 0; j < n; ++j) {
    float bm = -INFINITY;
    int bi = 0x7fffffff;
    for (int kb = s0; kb < s1; kb += (int)blockDim.x * 4) {
      float w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = kb + i * (int)blockDim.x + tid;
        w[i] = k < s1 ? f(j, k) : -INFINITY;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = kb + i * (int)blockDim.x + tid;
        if (k < s1 && (w[i] > bm || bi == 0x7fffffff)) { bm = w[i]; bi = k; }
      }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, bm, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (oi != 0x7fffffff && (bi == 0x7fffffff || om > bm || (om == bm && oi < bi))) { bm = om; bi = oi; }
    }
    if (lane == 0) { sc->amax[j][warp] = bm; sc->aidx[j][warp] = bi; }
  }
  __syncthreads();
  for (int j = warp; j < n; j += row_warps()) {
    const bool on = lane < row_warps();
    float bm = on ? sc->amax[j][lane] : -INFINITY;
    int bi = on ? sc->aidx[j][lane] : 0x7fffffff;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, bm, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (oi != 0x7fffffff && (bi == 0x7fffffff || om > bm || (om == bm && oi < bi))) { bm = om; bi = oi; }
    }
    if (lane < rs.C) { store_in_cta(&sc->gmax[j][rs.rank], lane, bm); store_in_cta(&sc->gidx[j][rs.rank], lane, bi); }
  }
  cluster_sync_all_threads();
  if (tid < n) {
    float bm = sc->gmax[tid][0];
    int bi = sc->gidx[tid][0];
    for (int c = 1; c < rs.C; ++c) {
      const float om = sc->gmax[tid][c];
      const int oi = sc->gidx[tid][c];
      if (oi != 0x7fffffff && (bi == 0x7fffffff || om > bm || (om == bm && oi < bi))) { bm = om; bi = oi; }
    }
    sc->arg[tid] = bi;
  }
  __syncthreads();
}

// The rejection rule (Sec. 2.1) for one sequence on a cluster: pv(j, k) / qv(j, k) = value k of the target's /
// draft's row j (qv unused when greedy), ids [gamma] draft ids (each already known to lie in [0, V)), ub
// [gamma+1] uniforms.  Exactly one CTA returns true, with the accepted count r and the next token.
template <class PV, class QV>
__device__ bool rule_rows(PV pv, QV qv, const int* ids, const float* ub, int gamma, int V, int greedy, const RowSlice& rs,
                          RowScratch* sc, int& r, int& tok) {
  if (greedy) {
    for (int j0 = 0;; j0 += ARG_ROWS) {
      const int n = min(ARG_ROWS, gamma + 1 - j0);
      rows_argmax([&](int j, int k) { return pv(j0 + j, k); }, n, V, rs, sc);
      for (int j = 0; j < n; ++j) {
        r = j0 + j;
        tok = sc->arg[j];
        if (r == gamma || tok != ids[r]) return rs.rank == 0;
      }
      cluster_sync_all_threads();   // the exchange buffers are written again
    }
  }
  if (threadIdx.x == 0) sc->first_reject = gamma;
  __syncthreads();
  for (int j = threadIdx.x; j < gamma; j += blockDim.x)   // the accept tests are independent
    if (!accept_test(ub[j], pv(j, ids[j]), qv(j, ids[j]))) atomicMin(&sc->first_reject, j);
  __syncthreads();
  r = sc->first_reject;
  const int rr = r;
  if (rr < gamma) return row_sample([&](int k) { return fmaxf(0.0f, __fsub_rn(pv(rr, k), qv(rr, k))); }, V, ub[gamma], rs, sc, tok);
  return row_sample([&](int k) { return pv(rr, k); }, V, ub[gamma], rs, sc, tok);
}

// The rejection rule on given probability rows: C CTAs per sequence.
__global__ void __launch_bounds__(ROW_THREADS)
reject_sample_kernel(const float* __restrict__ p, const float* __restrict__ q, const int* __restrict__ ids,
                     const float* __restrict__ u, int gamma, int V, int greedy, int C, int* __restrict__ n_acc,
                     int* __restrict__ next) {
  __shared__ RowScratch sc;
  const int b = blockIdx.x / C;
  const RowSlice rs = row_slice(C);
  const float* pb = p + (size_t)b * (gamma + 1) * V;
  const float* qb = q ? q + (size_t)b * gamma * V : nullptr;
  const int* idb = ids + (size_t)b * gamma;
  const float* ub = u ? u + (size_t)b * (gamma + 1) : nullptr;
  // a draft id outside [0, V) cannot index a row: the sequence is reported as n_acc = next = -1
  bool bad = false;
  for (int j = 0; j < gamma; ++j) bad |= (unsigned)idb[j] >= (unsigned)V;
  if (bad) {      // the same in every CTA of the cluster
    if (rs.rank == 0 && threadIdx.x == 0) { n_acc[b] = -1; next[b] = -1; }
    return;
  }
  int r, tok;
  const bool mine = rule_rows([&](int j, int k) { return pb[(size_t)j * V + k]; }, [&](int j, int k) { return qb[(size_t)j * V + k]; },
                              idb, ub, gamma, V, greedy, rs, &sc, r, tok);
  if (mine && threadIdx.x == 0) { n_acc[b] = r; next[b] = tok; }
}

}  // namespace spd
