// Dense linear maps on the 5th-generation tensor cores: Y[R][N] = X[R][K] W[N][K]^T for every
// projection of the prefill (Eq. 1 in one pass), of the batched steps and of the image adapter.
//
// The WEIGHTS are the M operand of tcgen05.mma (128 rows per CTA, 256 per CTA pair) and the
// activation rows the N operand, so the tile is cut to the number of rows there are: any R is
// ceil(R / BN) tiles of BN <= 256 rows, BN a multiple of 16, instead of multiples of 128.  The
// accumulator is Y^T: a lane of tensor memory is an output column, so a warp's stores of one
// activation row are consecutive addresses.
//
// Precision: X is an fp32 quantity given as two bf16 matrices hi + lo (x = hi + lo up to 2^-17 |x|);
// a ring stage holds the weight tile once and both activation tiles, and both products accumulate
// into the same fp32 columns.
//
// Roles of the 10 warps: 0 feeds TMA (128-byte swizzle, no multicast), 1 issues the MMAs, 2..9 read the
// accumulator back; two accumulators of 256 columns let a tile's epilogue run under the next tile's
// MMAs.  CG = 2: a CTA pair works on one 256-row weight tile, each CTA loads its own half of both
// operands, the even CTA issues (cta_group::2), which halves the activation bytes each SM reads.
//
// Work: persistent units (a CTA, or a pair) take the items u, u + U, ... of weight tiles x activation
// tiles x K slices, the activation tile fastest, so that the units that run at the same time share a
// weight tile (one fetch from HBM) and walk K in step (their requests for the same activation lines
// meet in L2: dealing every unit an equal run of K blocks instead, which puts the units at different
// K, measured 10-15 % slower although no wave was left partly empty).  With several slices, slice s
// leaves its partial product at out_f32 + s * R * ldo and the kernel that reads the result adds the
// slices up in order (deterministic).
//
// Dependent launch: the weights of the first ring stages are requested before the kernel waits for its
// predecessor in the stream, which hides the launch, the barrier set-up and the first HBM latency of
// a kernel that often runs for less than 10 us.
//
// 640 rows, us, against a kernel of 128 x 128 tiles with two CTAs per SM (gate/up: 67 -> 89 % of the measured cuBLAS
// rate on the largest): QKV 131 -> 95, O 57 -> 34, gate/up + SwiGLU 212 -> 159, down 133 -> 86.
#pragma once
#include <cuda.h>

#include "spd_device.cuh"

namespace spd {

constexpr int TC_BK = 64;          // columns of K per ring stage: one 128-byte swizzle row of bf16
constexpr int UG_EPI_WARPS = 8;      // two per 32-lane quarter of tensor memory, taking turns at 32-column pieces
constexpr int UG_THREADS = 64 + 32 * UG_EPI_WARPS;
constexpr int UG_BN_MAX = 256;
constexpr int UG_STAGES_MAX = 12;
constexpr int UG_SMEM = 225 * 1024;                       // ring + barriers: one CTA per SM
constexpr int UG_RING = UG_SMEM - 1024 - 512;             // minus alignment slack and barriers
constexpr int UG_A_BYTES = 128 * TC_BK * 2;

// K-major operand tile in shared memory, rows of 128 bytes, 128-byte swizzle: 8-row groups are
// 1024 bytes apart (stride byte offset), leading byte offset 1 (unused for swizzled K-major).
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
  return (uint64_t)((smem_addr >> 4) & 0x3FFFu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// GELU in its exact form x * Phi(x), the non-linearity between the two linear layers of the image
// adapter g_theta (Sec. 2.2, Appendix A.1; the paper does not name it, LLaVA's projector uses it).
__device__ __forceinline__ float gelu_exact(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// epilogues
enum : int { UG_F32 = 0,      // out_f32[m][n] = y
             UG_GELU = 1,     // out_hi / out_lo[m][n] = split(gelu(y))
             UG_SWIGLU = 2 }; // weight rows (gate_0, up_0, gate_1, ...): out_hi / out_lo[m][n/2] = split(silu(gate) * up)

struct UgArgs {
  int N, R, K;              // weight rows, activation rows, inner dimension
  int bn, n_at;             // activation rows per tile, number of such tiles
  int tiles, kb;            // weight tiles x activation tiles; 64-wide K blocks
  int stages, slices;       // ring depth; K slices (1: whole sums)
  long long ldo;
  float* out_f32;
  __nv_bfloat16 *out_hi, *out_lo;
  int* err;
};

struct UgWork {
  int wt, at, slice, kb0, kb1;   // weight tile, activation tile, K slice and its K blocks
};

// The work list of one unit; every role of the CTA walks the same list.
struct UgIter {
  int cur, end, step;
  __device__ __forceinline__ UgIter(const UgArgs& a, int unit, int units) : cur(unit), end(a.tiles * a.slices), step(units) {}
  __device__ __forceinline__ bool next(const UgArgs& a, UgWork& w) {
    if (cur >= end) return false;
    w.slice = cur / a.tiles;
    const int tile = cur - w.slice * a.tiles;
    w.wt = tile / a.n_at;
    w.at = tile - w.wt * a.n_at;
    w.kb0 = w.slice * a.kb / a.slices;
    w.kb1 = (w.slice + 1) * a.kb / a.slices;
    cur += step;
    return true;
  }
};

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

template <int CG>
__device__ __forceinline__ void ug_load(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  if constexpr (CG == 2)
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(0), "r"(bar) : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(0), "r"(bar) : "memory");
}
template <int CG>
__device__ __forceinline__ void ug_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  if constexpr (CG == 2)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"(acc) : "memory");
  else
    umma_bf16(d, ad, bd, idesc, acc);
}
// arrives (in both CTAs of a pair) once the MMAs issued so far have completed
template <int CG>
__device__ __forceinline__ void ug_commit(uint64_t* bar) {
  if constexpr (CG == 2)
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
  else
    umma_commit(bar);
}
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, unsigned parity, volatile int* err, int code) {
  for (unsigned it = 0; it < SPIN_LIMIT_MBAR; ++it) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((it & 1023u) == 1023u && *err != DEV_OK) return false;
  }
  atomicCAS(const_cast<int*>(err), DEV_OK, code);
  return false;
}

// 32 activation rows m0.. of output column n (this thread's lane) leave the accumulator.
template <int EPI>
__device__ __forceinline__ void ug_store(const UgArgs& a, float (&v)[32], int n, int m0, int mend, int lane, float* f32) {
  if constexpr (EPI == UG_F32) {
    if (n < a.N) {
      float* p = f32 + (long long)m0 * a.ldo + n;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (m0 + j < mend) p[j * a.ldo] = v[j];
    }
  } else {
    // neighbouring lanes (columns n, n ^ 1) trade values so that the even lane has both columns of row
    // m0 + 2q and the odd lane both columns of row m0 + 2q + 1
    const bool odd = lane & 1;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const float keep = odd ? v[2 * q + 1] : v[2 * q];
      const float got = __shfl_xor_sync(0xffffffffu, odd ? v[2 * q] : v[2 * q + 1], 1);
      const float c0 = odd ? got : keep, c1 = odd ? keep : got;   // columns n & ~1 and n | 1
      const int m = m0 + 2 * q + (odd ? 1 : 0);
      if (m < mend) {
        if constexpr (EPI == UG_SWIGLU) {
          if ((n | 1) < a.N) {
            const float x = (c0 / (1.0f + expf(-c0))) * c1;
            const __nv_bfloat16 h = __float2bfloat16_rn(x);
            const long long o = (long long)m * a.ldo + (n >> 1);
            a.out_hi[o] = h;
            a.out_lo[o] = __float2bfloat16_rn(x - __bfloat162float(h));
          }
        } else {
          const float x0 = gelu_exact(c0), x1 = gelu_exact(c1);
          const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
          const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __low2float(h), x1 - __high2float(h));
          const long long o = (long long)m * a.ldo + (n & ~1);
          if ((n | 1) < a.N) {           // ldo is a multiple of 8 here: 4-byte aligned pairs
            *reinterpret_cast<__nv_bfloat162*>(a.out_hi + o) = h;
            *reinterpret_cast<__nv_bfloat162*>(a.out_lo + o) = l;
          } else if ((n & ~1) < a.N) {
            a.out_hi[o] = __low2bfloat16(h);
            a.out_lo[o] = __low2bfloat16(l);
          }
        }
      }
    }
  }
}

template <int CG, int EPI>
__global__ void __cluster_dims__(CG, 1, 1) __launch_bounds__(UG_THREADS, 1)
umma_gemm_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_hi,
                 const __grid_constant__ CUtensorMap map_lo, const UgArgs a) {
  extern __shared__ uint8_t ug_smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ug_smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + UG_RING);
  uint64_t* empty = full + UG_STAGES_MAX;
  uint64_t* acc_full = empty + UG_STAGES_MAX;     // [2]
  uint64_t* acc_empty = acc_full + 2;             // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* err = a.err;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = CG == 2 ? (int)(blockIdx.x & 1) : 0;
  const int unit = blockIdx.x / CG, units = gridDim.x / CG;
  const int bn_cta = a.bn / CG;                                     // activation rows this CTA loads per tile
  const uint32_t b_bytes = (uint32_t)bn_cta * TC_BK * 2, stage_bytes = UG_A_BYTES + 2 * b_bytes;

  if (tid == 0) {
    for (int i = 0; i < a.stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], UG_EPI_WARPS * CG); }
    mbar_fence_init();
  }
  if (warp == 1) {
    if constexpr (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if constexpr (CG == 2) cluster_sync_all_threads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;

  pdl_trigger();
  UgIter iter(a, unit, units);
  UgWork w{};
  if (warp == 0) {
    // ---- TMA: this CTA's weight rows and its share of the activation rows; the even CTA's barrier counts
    // the bytes of both.  First the weights of a ring's worth of stages, then -- once the predecessor's
    // results are visible -- everything else.
    auto load_w = [&](int kb, int s) {
      if (rank == 0) mbar_arrive_expect_tx(&full[s], CG * stage_bytes);
      const uint32_t bar = CG == 2 ? cluster_map(smem_u32(&full[s]), 0) : smem_u32(&full[s]);
      ug_load<CG>(smem_u32(ring) + s * stage_bytes, &map_w, kb * TC_BK, (w.wt * CG + rank) * 128, bar);
    };
    auto load_x = [&](int kb, int s) {
      const uint32_t bar = CG == 2 ? cluster_map(smem_u32(&full[s]), 0) : smem_u32(&full[s]);
      const uint32_t dst = smem_u32(ring) + s * stage_bytes + UG_A_BYTES;
      const int arow = w.at * a.bn + rank * bn_cta;
      ug_load<CG>(dst, &map_hi, kb * TC_BK, arow, bar);
      ug_load<CG>(dst + b_bytes, &map_lo, kb * TC_BK, arow, bar);
    };
    int ahead = 0;
    {
      UgIter first = iter;
      while (ahead < a.stages && first.next(a, w))
        for (int kb = w.kb0; kb < w.kb1 && ahead < a.stages; ++kb, ++ahead)
          if (elect_one()) load_w(kb, ahead);
    }
    __syncwarp();
    pdl_wait();
    int s = 0, i = 0;
    unsigned ph = 0;
    bool ok = true;
    while (ok && iter.next(a, w)) {
      for (int kb = w.kb0; kb < w.kb1; ++kb, ++i) {
        if (i < ahead) {
          if (elect_one()) load_x(kb, s);
        } else {
          ok = mbar_wait_cluster(&empty[s], ph ^ 1u, err, DEV_TIMEOUT_EMPTY);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (elect_one()) { load_w(kb, s); load_x(kb, s); }
        }
        __syncwarp();
        if (++s == a.stages) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ---- MMAs (one CTA of a pair issues for both)
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.bn >> 3) << 17) | ((uint32_t)(128 * CG >> 4) << 24);
      int s = 0, buf = 0;
      unsigned ph = 0, aph = 0;
      bool ok = true;
      while (ok && iter.next(a, w)) {
        ok = mbar_wait_cluster(&acc_empty[buf], aph ^ 1u, err, DEV_TIMEOUT_EMPTY);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem_base + (uint32_t)buf * UG_BN_MAX;
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          ok = mbar_wait_cluster(&full[s], ph, err, DEV_TIMEOUT_FULL);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = smem_u32(ring) + s * stage_bytes;
          const uint64_t wd = umma_desc(st), hd = umma_desc(st + UG_A_BYTES), ld = umma_desc(st + UG_A_BYTES + b_bytes);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k) {
              ug_mma<CG>(d, wd + 2 * k, hd + 2 * k, idesc, (kb > w.kb0 || k > 0) ? 1u : 0u);
              ug_mma<CG>(d, wd + 2 * k, ld + 2 * k, idesc, 1u);
            }
            ug_commit<CG>(&empty[s]);
            if (kb + 1 == w.kb1) ug_commit<CG>(&acc_full[buf]);
          }
          __syncwarp();
          if (++s == a.stages) { s = 0; ph ^= 1u; }
        }
        if (buf) aph ^= 1u;
        buf ^= 1;
      }
    }
  } else {
    // ---- epilogue: warp reads TMEM lanes 32 (warp & 3) .. + 31 = weight rows of this CTA's tile
    pdl_wait();
    const int row = (warp & 3) * 32 + lane, part = (warp - 2) >> 2;
    int buf = 0;
    unsigned aph = 0;
    while (iter.next(a, w)) {
      const int n = (w.wt * CG + rank) * 128 + row;
      const int m_first = w.at * a.bn, mend = min(a.R, m_first + a.bn);
      bool ok = mbar_wait_cluster(&acc_full[buf], aph, err, DEV_TIMEOUT_FULL);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t tbase = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)buf * UG_BN_MAX;
      float* f32 = EPI == UG_F32 ? a.out_f32 + (long long)w.slice * a.R * a.ldo : nullptr;
#pragma unroll 1
      for (int c0 = part * 32; c0 < mend - m_first; c0 += 32 * (UG_EPI_WARPS / 4)) {
        uint32_t raw[32];
        tmem_ld32(tbase + (uint32_t)c0, raw);
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(raw[j]);
        ug_store<EPI>(a, v, n, m_first + c0, mend, lane, f32);
      }
      // the accumulator is free: the issuing CTA may start the tile after next in it
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(CG == 2 ? cluster_map(smem_u32(&acc_empty[buf]), 0) : smem_u32(&acc_empty[buf]));
      if (buf) aph ^= 1u;
      buf ^= 1;
    }
  }
  pdl_wait();     // (no effect where it was called above) nothing of this CTA ends before its predecessor has
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*err != DEV_OK) for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
  if constexpr (CG == 2) cluster_sync_all_threads();
  if (warp == 1) {
    if constexpr (CG == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
}

}  // namespace spd
