// Top-k / top-p (nucleus) truncation of probability rows ahead of the speculative-sampling rule.
// The paper decodes greedily and names sampling with top-p / top-k as future work (Sec. 4
// "Decoding"); truncating and renormalising BOTH the target's and the draft's rows and applying
// the unchanged rule of Sec. 2.1 to them keeps the method's guarantee for the truncated target
// distribution.
//
// Definitions (exact, so that the result does not depend on the order of any reduction):
//   order  larger probability first, lower index first among equal probabilities;
//   mass   W_i = trunc(w_i * 2^32), summed as integers;
//   top-k  the first k tokens of the order;
//   top-p  among the kept tokens (total mass Z) the shortest prefix of the order whose mass
//          reaches T = ceil(Z * trunc(top_p * 2^24) / 2^24), at least one token;
//   output w_i / S for kept tokens with S = float(kept mass) * 2^-32, 0 for the others.
// One CTA of 1024 threads per row, the row in shared memory and never changed: a cut is a value and an
// index (kept: larger values, and values equal to it up to that index).  The cut value is found digit by
// digit over the fp32 bit patterns (monotone for non-negative values) with a histogram of counts
// (top-k) or masses (top-p); ties are resolved in index order only when some of them are dropped.
// Bin totals are kept as two 32-bit sums (low 16 bits, the rest), which 32-bit shared-memory atomics add
// exactly.
//
// Bound by shared-memory atomics of the first digit: probabilities share a handful of exponents.  2048
// bins (11 bits: eight to an exponent) spread them; 256 bins where the row leaves no room for more.
// 11 rows x 32000, k 50, p 0.9: 98 us with 256 threads, four 8-bit digits and a marked row; 33 us this way.
#pragma once
#include "spd_sample.cuh"

namespace spd {

constexpr int TRUNC_THREADS = 1024, TRUNC_WARPS = 32;
constexpr int TRUNC_BINS = 2048, TRUNC_BINS_MIN = 256;

template <int BINS>
struct TruncScratch {
  unsigned int hlo[BINS], hhi[BINS];   // per-bin totals as sum(v & 0xffff) and sum(v >> 16): 32-bit atomics, exact 64-bit result
  unsigned long long wred[TRUNC_WARPS];
  unsigned int wcnt[TRUNC_WARPS];
  unsigned long long rem;   // count or mass still to be taken at the current digit
  unsigned long long bin;   // total of the chosen bin
  unsigned int chosen;
  int last;
};

struct Cut {
  float value;
  int last;                 // of the entries equal to `value`, those up to this index are kept
  __device__ __forceinline__ bool keeps(float w, int i) const { return w > value || (w == value && i <= last); }
};

template <int BINS>
__device__ __forceinline__ unsigned long long trunc_sum(unsigned long long v, TruncScratch<BINS>* sc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) sc->wred[warp] = v;
  __syncthreads();
  v = sc->wred[lane];
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Finds the bin in which the running total from the top bin downwards crosses sc->rem: leaves it in
// sc->chosen with its total in sc->bin, and reduces sc->rem to what is still needed inside it.
template <int BINS>
__device__ void pick_bin(TruncScratch<BINS>* sc) {
  constexpr int PER = BINS > TRUNC_THREADS ? BINS / TRUNC_THREADS : 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned long long h[PER], mine = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int b = tid * PER + i;
    h[i] = b < BINS ? ((unsigned long long)sc->hhi[b] << 16) + sc->hlo[b] : 0ull;
    mine += h[i];
  }
  // totals of the bins above this thread's: suffix scan inside the warp, then across warps
  unsigned long long incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += t;
  }
  if (lane == 0) sc->wred[warp] = incl;
  __syncthreads();
  unsigned long long tot = sc->wred[lane], up = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_down_sync(0xffffffffu, up, o);
    if (lane + o < 32) up += t;
  }
  unsigned long long above = incl - mine + __shfl_sync(0xffffffffu, up - tot, warp);
  const unsigned long long rem = sc->rem;
  __syncthreads();
#pragma unroll
  for (int i = PER - 1; i >= 0; --i) {
    if (h[i] > 0 && above < rem && rem <= above + h[i]) { sc->chosen = (unsigned)(tid * PER + i); sc->rem = rem - above; sc->bin = h[i]; }
    above += h[i];
  }
  __syncthreads();
}

// The cut that keeps the first entries of the order (among those `had` keeps) until `target` is reached (MASS:
// their mass, else their number).  Requires 1 <= target <= total of the entries still kept.
template <bool MASS, int BINS>
__device__ Cut find_cut(const float* row, int V, const Cut& had, unsigned long long target, TruncScratch<BINS>* sc) {
  constexpr int BITS = BINS == 2048 ? 11 : 8;
  static_assert(BINS == (1 << BITS), "");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned int prefix = 0;
  if (tid == 0) sc->rem = target;
  int shift = 31;                        // the sign bit is 0: 31 bits to go
  while (shift > 0) {
    const int width = shift < BITS ? shift : BITS, top = shift;
    shift -= width;
    const unsigned int mask = (1u << width) - 1u;
    for (int b = tid; b < BINS; b += TRUNC_THREADS) { sc->hlo[b] = 0; sc->hhi[b] = 0; }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < V; i += TRUNC_THREADS) {
      const float w = row[i];
      const unsigned int bits = __float_as_uint(w);
      if (((bits ^ prefix) >> top) != 0 || !had.keeps(w, i)) continue;
      const unsigned int b = (bits >> shift) & mask;
      if (MASS) {
        const unsigned long long v = to_fixed(w);
        atomicAdd(&sc->hlo[b], (unsigned)(v & 0xffffull));
        atomicAdd(&sc->hhi[b], (unsigned)(v >> 16));
      } else {
        atomicAdd(&sc->hlo[b], 1u);
      }
    }
    __syncthreads();
    pick_bin(sc);
    prefix |= sc->chosen << shift;
  }
  // prefix = bit pattern of the cut value; rem = count / mass still needed from the entries equal to it
  Cut cut{__uint_as_float(prefix), V};
  unsigned long long need = sc->rem, have = sc->bin;
  if (MASS) {
    const unsigned long long wc = to_fixed(cut.value);
    need = wc ? (need + wc - 1) / wc : 0xffffffffull;
    have = wc ? have / wc : 0;
  }
  if (need >= have) return Cut{cut.value, had.value == cut.value ? had.last : V};   // all of them
  // the need-th equal entry in index order; warp w looks at a contiguous piece
  const int VW = (((V + TRUNC_WARPS - 1) / TRUNC_WARPS) + 31) & ~31, k0 = min(V, warp * VW), k1 = min(V, k0 + VW);
  unsigned int mine = 0;
  for (int k = k0; k < k1; k += 32) {
    const int i = k + lane;
    mine += __popc(__ballot_sync(0xffffffffu, i < k1 && row[i] == cut.value && had.keeps(row[i], i)));
  }
  if (lane == 0) sc->wcnt[warp] = mine;
  __syncthreads();
  unsigned int before = 0;
  for (int w = 0; w < warp; ++w) before += sc->wcnt[w];
  if (before < need && need <= (unsigned long long)before + mine) {
    for (int k = k0; k < k1; k += 32) {
      const int i = k + lane;
      const unsigned int eq = __ballot_sync(0xffffffffu, i < k1 && row[i] == cut.value && had.keeps(row[i], i));
      if (before + __popc(eq) >= need) {
        const int n = (int)need - (int)before;        // the n-th set bit
        if (((eq >> lane) & 1u) && __popc(eq & ((2u << lane) - 1u)) == n) sc->last = i;
        break;
      }
      before += __popc(eq);
    }
  }
  __syncthreads();
  cut.last = sc->last;
  return cut;
}

template <int BINS>
__global__ void __launch_bounds__(TRUNC_THREADS)
truncate_rows_kernel(const float* __restrict__ in, float* __restrict__ out, int V, int top_k, float top_p) {
  extern __shared__ float trunc_row[];
  __shared__ TruncScratch<BINS> sc;
  const float* src = in + (size_t)blockIdx.x * V;
  float* dst = out + (size_t)blockIdx.x * V;
#pragma unroll 8
  for (int i = threadIdx.x; i < V; i += TRUNC_THREADS) {
    const float w = src[i];
    trunc_row[i] = w > 0.0f ? w : 0.0f;
  }
  __syncthreads();
  Cut cut{0.0f, V};                      // everything (entries are >= 0)
  if (top_k >= 1 && top_k < V) cut = find_cut<false>(trunc_row, V, cut, (unsigned long long)top_k, &sc);
  auto mass = [&]() {
    unsigned long long z = 0;
#pragma unroll 4
    for (int i = threadIdx.x; i < V; i += TRUNC_THREADS) {
      const float w = trunc_row[i];
      if (cut.keeps(w, i)) z += to_fixed(w);
    }
    return trunc_sum(z, &sc);
  };
  unsigned long long z = mass();
  if (top_p > 0.0f && top_p < 1.0f && z > 0) {
    const unsigned long long p24 = static_cast<unsigned long long>(__fmul_rn(top_p, 16777216.0f));
    unsigned long long T = (z * p24 + 16777215ull) >> 24;
    if (T < 1) T = 1;
    cut = find_cut<true>(trunc_row, V, cut, T, &sc);
    z = mass();
  }
  const float S = __fmul_rn(__ull2float_rn(z), 2.3283064365386963e-10f);   // * 2^-32, exact
#pragma unroll 4
  for (int i = threadIdx.x; i < V; i += TRUNC_THREADS) {
    const float w = trunc_row[i];
    dst[i] = cut.keeps(w, i) ? (z ? __fdiv_rn(w, S) : w) : 0.0f;
  }
}

}  // namespace spd
