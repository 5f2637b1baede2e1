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
// cluster barrier per draw (about 1 us with the launch of the cluster; one CTA spares it).  Bound by latency: the
// ids, the two values of every test, the row, the search, one after the other, and few instructions to fetch: a search
// unrolled over 16 steps of 32 entries took 3200 cycles of a draw from 1000 weights, narrowing 32-fold at a time 900.
// Device time of the rule on one sequence, 6 rows not in L2, sampled, us: 1000 entries 3.5 (with clusters, a barrier more and the
// unrolled search 5.4; one CTA of 256 threads and a serial walk 4.0), 32000 entries 6.4 (8.4; 28).
constexpr int ROW_THREADS = 1024, ROW_WARPS = ROW_THREADS / 32, ROW_CTAS_MAX = 8;
__device__ __forceinline__ int row_warps() { return (int)(blockDim.x >> 5); }
constexpr int ARG_ROWS = 8;     // rows whose arg-max is taken together
constexpr int RULE_MANY = 8;    // sequences from which on a greedy rule takes all its rows at once

struct RowScratch {
  unsigned long long wsum[ROW_WARPS];
  unsigned long long tot[ROW_CTAS_MAX];            // every CTA's mass
  unsigned amax[ARG_ROWS][ROW_WARPS];                 // arg-max of several rows at once
  int aidx[ARG_ROWS][ROW_WARPS];
  unsigned gmax[ARG_ROWS][ROW_CTAS_MAX];
  int gidx[ARG_ROWS][ROW_CTAS_MAX];
  int arg[ARG_ROWS];
  int result;
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

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {   // three 32-bit sums of 27-bit parts
  return (unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)(v & 0x7ffffffull)) +
         ((unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)((v >> 27) & 0x7ffffffull)) << 27) +
         ((unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)(v >> 54)) << 54);
}

// What a row's draws need: the row's total mass (the same in every CTA) and, of this CTA's warps, the mass
// of warp `lane` and of all up to it.
struct RowMass {
  unsigned long long Z, own, upto;
};

// Masses of the row's weights; emit(k, w) sees every weight of this CTA's slice once.  The weights can then be
// drawn from with row_pick.  (A second call needs a barrier between them: the scratch is written again.)
template <class WF, class EM>
__device__ RowMass row_mass(WF wf, EM emit, int V, const RowSlice& rs, RowScratch* sc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int k0, k1;
  row_piece(rs, V, warp, k0, k1);
  unsigned long long s = 0;
  for (int kb = k0; kb < k1; kb += 32 * ROW_UNROLL) {
    float w[ROW_UNROLL];
#pragma unroll
    for (int i = 0; i < ROW_UNROLL; ++i) {
      const int k = kb + i * 32 + lane;
      w[i] = k < k1 ? wf(k) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < ROW_UNROLL; ++i) {
      const int k = kb + i * 32 + lane;
      if (k < k1) {
        s += to_fixed(w[i]);
        emit(k, w[i]);
      }
    }
  }
  s = warp_sum(s);
  if (lane == 0) sc->wsum[warp] = s;
  __syncthreads();
  RowMass m;
  m.own = m.upto = lane < row_warps() ? sc->wsum[lane] : 0ull;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, m.upto, o);
    if (lane >= o) m.upto += t;
  }
  m.Z = __shfl_sync(0xffffffffu, m.upto, 31);
  if (rs.C > 1) {
    if (warp == 0 && lane < rs.C) store_in_cta(&sc->tot[rs.rank], lane, m.Z);
    cluster_sync_all_threads();
    m.Z = 0;
    for (int c = 0; c < rs.C; ++c) m.Z += sc->tot[c];
  }
  return m;
}

// Arg-max (lowest index on ties) of n <= ARG_ROWS rows at once: f(j, k) = value k of row j; the results are
// left in sc->arg of every CTA.  A warp takes a piece of one row, so that all rows' loads travel together: 6 x 32000 on
// a cluster of 8 in 7.5 us, 9.5 with the rows one after the other and all warps on each.
template <class F>
__device__ void rows_argmax(F f, int n, int V, const RowSlice& rs, RowScratch* sc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = row_warps();
  const int VC = (V + rs.C - 1) / rs.C, s0 = min(V, rs.rank * VC), s1 = min(V, s0 + VC);
  const int P = n < nw ? nw / n : 1, VP = (((s1 - s0 + P - 1) / P) + 31) & ~31;
  // a value as an unsigned number of the same order (-0 as 0, a NaN below everything)
  auto key = [](float v) {
    const unsigned b = __float_as_uint(v + 0.0f);
    return v != v ? 0u : (b & 0x80000000u ? ~b : b | 0x80000000u);
  };
  // largest value of the warp, lowest index on ties (0x7fffffff: no entry)
  auto reduce = [&](unsigned& bk, int& bi) {
    const unsigned top = __reduce_max_sync(0xffffffffu, bk);
    bi = (int)__reduce_min_sync(0xffffffffu, bk == top ? (unsigned)bi : 0x7fffffffu);
    bk = top;
  };
  for (int item = warp; item < n * P; item += nw) {
    const int j = item / P, pc = item - j * P, k0 = min(s1, s0 + pc * VP), k1 = min(s1, k0 + VP);
    float bm = -INFINITY;
    int bi = 0x7fffffff;
    for (int kb = k0; kb < k1; kb += 32 * ROW_UNROLL) {
      float w[ROW_UNROLL];
#pragma unroll
      for (int i = 0; i < ROW_UNROLL; ++i) {
        const int k = kb + i * 32 + lane;
        w[i] = k < k1 ? f(j, k) : -INFINITY;
      }
#pragma unroll
      for (int i = 0; i < ROW_UNROLL; ++i) {
        const int k = kb + i * 32 + lane;
        if (k < k1 && (w[i] > bm || bi == 0x7fffffff)) { bm = w[i]; bi = k; }
      }
    }
    unsigned bk = bi == 0x7fffffff ? 0u : key(bm);
    reduce(bk, bi);
    if (lane == 0) { sc->amax[j][pc] = bk; sc->aidx[j][pc] = bi; }
  }
  __syncthreads();
  for (int j = warp; j < n; j += nw) {
    unsigned bk = lane < P ? sc->amax[j][lane] : 0u;
    int bi = lane < P ? sc->aidx[j][lane] : 0x7fffffff;
    reduce(bk, bi);
    if (rs.C == 1) {
      if (lane == 0) sc->arg[j] = bi;
    } else if (lane < rs.C) {
      store_in_cta(&sc->gmax[j][rs.rank], lane, bk);
      store_in_cta(&sc->gidx[j][rs.rank], lane, bi);
    }
  }
  if (rs.C > 1) {
    cluster_sync_all_threads();
    if (tid < n) {
      unsigned bk = sc->gmax[tid][0];
      int bi = sc->gidx[tid][0];
      for (int c = 1; c < rs.C; ++c) {      // (slices in order: the first of equals has the lowest index)
        const unsigned ok = sc->gmax[tid][c];
        const int oi = sc->gidx[tid][c];
        if (oi != 0x7fffffff && (bi == 0x7fffffff || ok > bk)) { bk = ok; bi = oi; }
      }
      sc->arg[tid] = bi;
    }
  }
  __syncthreads();
}

// The token that uniform u draws from the weights of the preceding row_mass.  Exactly one CTA of the
// cluster, the one whose slice holds the token, returns true.
template <class WF>
__device__ bool row_pick(WF wf, int V, const RowMass& m, float u, const RowSlice& rs, RowScratch* sc, int& tok) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (m.Z == 0) {      // no mass at all: the largest weight, lowest index on ties; entries that are no numbers last
    rows_argmax([&](int, int k) { const float w = wf(k); return w > -1.0f ? w : -1.0f; }, 1, V, rs, sc);
    tok = sc->arg[0];
    cluster_sync_all_threads();   // (the exchange buffers may be used again)
    return rs.rank == 0;
  }
  const unsigned long long T = threshold(m.Z, u);
  unsigned long long base = 0;
  if (rs.C > 1) {
    int cc = 0;
    while (cc < rs.C - 1 && T >= base + sc->tot[cc]) base += sc->tot[cc++];
    if (cc != rs.rank) return false;
  }
  // the warp whose piece the running total crosses T in
  const unsigned over = __ballot_sync(0xffffffffu, T < base + m.upto);
  const int ww = over ? __ffs(over) - 1 : row_warps() - 1;
  base += __shfl_sync(0xffffffffu, m.upto - m.own, ww);
  if (warp == ww) {
    // narrowed 32-fold at a time: a lane sums a run of entries, the lane whose run the total crosses T in is next
    int k0, k1;
    row_piece(rs, V, warp, k0, k1);
    int len = k1 - k0;
    while (true) {
      const int run = (len + 31) >> 5, b0 = min(k1, k0 + lane * run), b1 = min(min(k1, k0 + len), b0 + run);
      unsigned long long own = 0;
#pragma unroll 4
      for (int k = b0; k < b1; ++k) own += to_fixed(wf(k));
      unsigned long long upto = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += t;
      }
      const unsigned past = __ballot_sync(0xffffffffu, T < base + upto && b0 < b1);
      const int l = past ? __ffs(past) - 1 : 0;
      base += __shfl_sync(0xffffffffu, upto - own, l);
      k0 += l * run;
      if (run <= 1) break;
      len = min(len - l * run, run);
    }
    const int found = max(min(k0, k1 - 1), 0);
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
  const RowMass m = row_mass(wf, [](int, float) {}, V, rs, sc);
  return row_pick(wf, V, m, u, rs, sc, tok);
}

// The rejection rule (Sec. 2.1) for one sequence on a cluster: pv(j, k) / qv(j, k) = value k of the target's /
// draft's row j (qv unused when greedy), ids [gamma] draft ids (each already known to lie in [0, V)), ub
// [gamma+1] uniforms; `rows`: the sequences of the launch.  Exactly one CTA returns true, with the accepted count r
// and the next token.
template <class PV, class QV>
__device__ bool rule_rows(PV pv, QV qv, const int* ids, const float* ub, int gamma, int V, int greedy, const RowSlice& rs,
                          RowScratch* sc, int rows, int& r, int& tok) {
  if (greedy) {
    // Few sequences: the first row alone, then the others together, as a draft that is off mostly is so at once.  One sequence,
    // 32000 entries on 8 CTAs, first token rejected / most accepted, us: 4.7 / 11.8, all rows together 9.4 / 9.7, row by row on one
    // CTA 6.2 / 53.  Of many sequences one gets further nearly always, and the launch lasts as long as the longest: together
    // (32 sequences 14.5 instead of 16.9).
    for (int j0 = 0, n = rows < RULE_MANY ? 1 : min(ARG_ROWS, gamma + 1);; j0 += n, n = min(ARG_ROWS, gamma + 1 - j0)) {
      rows_argmax([&](int j, int k) { return pv(j0 + j, k); }, n, V, rs, sc);
      for (int j = 0; j < n; ++j) {
        r = j0 + j;
        tok = sc->arg[j];
        if (r == gamma || tok != ids[r]) return rs.rank == 0;
      }
      cluster_sync_all_threads();   // the exchange buffers are written again
    }
  }
  // the accept tests are independent; every warp makes all of them, which spares two barriers
  r = gamma;
  for (int j0 = 0; j0 < gamma && r == gamma; j0 += 32) {
    const int j = j0 + (threadIdx.x & 31);
    const unsigned rej = __ballot_sync(0xffffffffu, j < gamma && !accept_test(ub[j], pv(j, ids[j]), qv(j, ids[j])));
    if (rej) r = j0 + __ffs(rej) - 1;
  }
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
  for (int j = threadIdx.x & 31; j < gamma; j += 32) bad |= (unsigned)idb[j] >= (unsigned)V;
  if (__any_sync(0xffffffffu, bad)) {      // the same in every CTA of the cluster
    if (rs.rank == 0 && threadIdx.x == 0) { n_acc[b] = -1; next[b] = -1; }
    return;
  }
  int r, tok;
  const bool mine = rule_rows([&](int j, int k) { return pb[(size_t)j * V + k]; }, [&](int j, int k) { return qb[(size_t)j * V + k]; },
                              idb, ub, gamma, V, greedy, rs, &sc, gridDim.x / C, r, tok);
  if (mine && threadIdx.x == 0) { n_acc[b] = r; next[b] = tok; }
}

}  // namespace spd
