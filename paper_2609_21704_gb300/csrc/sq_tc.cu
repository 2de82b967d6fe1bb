// sq_tc.cu -- tensor-core (tcgen05 / TMEM) linear layer (skinny GEMM, M rows
// padded to a multiple of 16 on the MMA's N side).
//
// Sec. III-D.3: the verify pass scores B * (K+1) rows at once (the draft
// pass B rows).  sq_linear_ex sends every call of more than 16 rows here, and from
// 3 to 16 rows the formats and shapes where this path measured faster than the
// streaming engine and the CUDA-core GEMV (rows past M are zero-filled by the TMA
// load).  Swap-AB: the weight tile is the MMA's A operand (M_mma = 128 weight rows), the activations are B (N_mma = NB, the
// activation rows padded to a multiple of 16), D = 128 x NB fp32 in TMEM:
//     D[n, m] = sum_k W[n, k] * x[m, k]   ->   y[m, n]
// Both operands are K-major fp16 tiles of 64 k (128 bytes per row) loaded by
// 2-D TMA with 128-byte swizzle into a ring of shared-memory stages; warp 0
// lane 0 issues the TMA copies, warp 1 lane 0 issues tcgen05.mma (4 x K16
// per stage) and commits each stage back to the producer; the epilogue warps,
// from warp 2 on, read the accumulator with tcgen05.ld (two warps share a 32-lane
// TMEM sub-partition and alternate blocks of its columns; up to 16 FP16 rows one
// has them all) and run the epilogue.  With the fused SiLU gate the CTA also loads the up
// rows' tile and accumulates a second NB-column block of TMEM.
//
// FP8 and INT4 weights: TMA brings the code tiles instead, and the eight
// epilogue warps (idle until the accumulator is final) dequantise each stage
// into the swizzled fp16 A tile (generic stores, fence.proxy.async, then an
// mbarrier arrive that releases the stage to the MMA thread).  FP8: exact
// E4M3 -> fp16, the per-row scale applied in the epilogue (exact).  INT4:
// c * s rounded once to fp16 (c exact, s the fp16 group scale), a relative
// rounding of at most 2^-11 per weight, far inside the linear layers' 1e-3
// relative-L2 tolerance (the per-(row, group) scale cannot be factored out
// of an MMA that accumulates over several groups).
//
// Split-K: the S CTAs of a cluster take consecutive K ranges of the same
// weight tile; each pushes its fp32 partials from TMEM to the shared memory of
// the CTA that finishes their column, and after a cluster barrier CTA r adds the
// S partials of its columns (about M / S consecutive ones) in rank order, so the
// result does not depend on timing.  Every mbarrier wait is bounded (a wait
// that gives up sets SQ_DEV_TIMEOUT and is skipped from then on), so every
// thread always reaches the cluster barriers.  After a wait gives up, the
// TMA producer requests nothing more and waits (bounded) for the copies it
// still has in flight, the MMA issuer issues nothing more, and the epilogue
// waits (bounded) on the commit that tracks every MMA issued before it
// reads TMEM and the allocation is released; the tile's results are then
// invalid and the status bit says so.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "sq_internal.h"

namespace sq {

static __device__ unsigned int g_tc_status;

constexpr int kTcBM = 128;      // weight rows per tile (MMA M)
constexpr int kTcBK = 64;       // k per stage: 64 fp16 = one 128-byte swizzle row
// Warp roles: warp 0 TMA, warp 1 MMA + TMEM, the EW others the epilogue (one or
// two per TMEM sub-partition) and, for quantised weights, the conversion of every
// stage before it (two per SM sub-partition, so that one's dependent chain hides
// behind the other's).  What follows the last MMA is latency bound (TMEM loads, the
// gate's exponential and quotient, the partials), so warps hide it: FP16 weights,
// four such warps -> eight, four layers (28 at 1.5B) per pass: 14B at 256 rows 817
// -> 682 us, at 80 rows (and lm_head) 794 -> 759; 7B at 256 1182 -> 963; 1.5B at
// 256 3576 -> 2529.  Up to 16 rows (FP16) a sub-partition has one block of
// columns, and four warps leave registers to the next launch's CTA: 28 layers of
// 1.5B at 16 rows 802 -> 795, a 1.5B decoder pass of three tokens 1318 -> 1314.
constexpr int tc_threads(int ew) { return 64 + 32 * ew; }
constexpr int kTcStageA = kTcBM * kTcBK * 2;  // 16 KB
// CTAs per cluster along K: up to 16 (non-portable cluster size, allowed at
// launch); the INT4 search keeps to the portable 8 it was measured at.
constexpr int kTcMaxSplit = 16;
constexpr int kTcMaxSplitInt4 = 8;

// ---------------------------------------------------------------- PTX

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor of a K-major tile with 128-byte swizzle:
// start address >> 4, leading byte offset 16 (unused by this layout), stride
// byte offset 1024 (one 8-row swizzle atom), descriptor version 1, swizzle
// mode 2 (128 B).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ void tc_mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                           uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.u32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// Stores to the shared memory of CTA `rank` of the cluster at the place where
// `addr` (a shared address) lies in this CTA's.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
  return remote;
}
__device__ __forceinline__ void st_dsmem_f32(uint32_t remote, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
}

// ---------------------------------------------------------------- kernel

struct TcArgs {
  const void* scales;  // FP8: fp32 [rows]; INT4: fp16 [rows, K/128]; FP16: unused
  int M;            // activation rows present
  int NB;           // MMA N: a CTA's activation rows rounded up to 16
  int colblocks;    // CTAs (grid z) that share a weight tile, NB activation rows each
  int64_t N;        // output columns (weight rows, or gate rows with SILU)
  int64_t K;
  int epi;
  int ksteps;       // ceil(K / 64)
  int splits;       // CTAs per cluster along K
  int nstages;
  int tmem_cols;
  uint32_t idesc;
  int stage_bytes;  // A (+ A_up) + B, multiple of 1024
  int b_off;        // offset of B inside a stage
  int c_off;        // offset of the code tiles inside a stage (FP8 / INT4)
  int c_bytes;      // bytes of one code tile
  int sc_off;       // INT4: byte offset of the CTA's group-scale block
  int sc_ng;        // INT4: groups per row held in the block (>= any CTA's need)
  int sc_bytes;     // INT4: bytes of the block
  int max_split;    // largest split-K factor whose partial tile fits in the stages
  int part_off;     // partial tile of a split: beside the stages, or 0: over them
  int two_per_sm;   // stages sized so that two CTAs share an SM
  int int4_large;   // INT4 weights of 20 MB and more at few rows: power-of-two split rule
  const __half* bias;
  const __half* residual;
  __half* y;
};

// WK: 0 fp16 weights, 1 INT4 codes, 2 FP8 codes (the GEMV family's numbering).
// CB: column blocks (instances of their own: the offsets cost the others up to
// 1.8 %).  EW: epilogue warps.
template <int WK, bool SILU, bool CB, int EW>
__global__ void __launch_bounds__(tc_threads(EW), 1)
    tc_linear_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tx,
                     const TcArgs a) {
  constexpr bool QUANT = WK != 0;
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment for the swizzle atoms
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  // a ring of stages [A (gate, up) | B | codes (gate, up; quantised only)]:
  // TMA brings B and either the fp16 A tiles or the code tiles, which the
  // converter warps dequantise into the stage's A tiles
  uint8_t* stages = smem;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)a.nstages * a.stage_bytes);
  uint64_t* full = bars;                       // stage landed (TMA)
  uint64_t* empty = bars + a.nstages;          // stage free again (MMA commit)
  uint64_t* accf = bars + 2 * a.nstages;       // accumulator final
  uint64_t* conv = bars + 2 * a.nstages + 1;   // A tiles converted (quantised)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 3 * a.nstages + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = a.splits;
  const uint32_t rank = S > 1 ? cluster_rank() : 0u;
  const int64_t tile = blockIdx.y;
  const int m0 = CB ? (int)blockIdx.z * a.NB : 0;  // this CTA's first activation row
  const int k_begin = (int)(((int64_t)rank * a.ksteps) / S);
  const int k_end = (int)(((int64_t)(rank + 1) * a.ksteps) / S);
  const int nk = k_end - k_begin;

  if (tid == 0) {
    for (int s = 0; s < a.nstages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&conv[s], EW);
    }
    mbar_init(accf, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (S > 1 && a.part_off) cluster_arrive();
  griddep_launch_dependents();

  bool timed_out = false;
  if (warp == 0) {
    if (lane == 0) {
      // --------------------------------------------------------- producer
      const uint32_t bytes =
          (uint32_t)((QUANT ? a.c_bytes : kTcStageA) * (SILU ? 2 : 1) + a.NB * 128);
      // weight tiles land in A (fp16) or in the stage's code area (quantised)
      const int wdst = QUANT ? a.c_off : 0;
      const int wdst_up = QUANT ? a.c_off + a.c_bytes : kTcStageA;
      // TMA x coordinate of a weight tile: k (fp16, FP8 bytes) or k / 2 (INT4 bytes)
      auto wx = [&](int k0) { return WK == 1 ? k0 / 2 : k0; };
      const int pre = nk < a.nstages ? nk : a.nstages;
      // weights never depend on the previous kernel: start them first
      for (int it = 0; it < pre; ++it) {
        uint8_t* st = stages + (size_t)it * a.stage_bytes;
        const int k0 = (k_begin + it) * kTcBK;
        mbar_arrive_expect_tx(&full[it], bytes);
        tma_load_2d(st + wdst, &tw, wx(k0), (int)(tile * kTcBM), &full[it]);
        if (SILU) tma_load_2d(st + wdst_up, &tw, wx(k0), (int)(a.N + tile * kTcBM), &full[it]);
      }
      griddep_wait();
      for (int it = 0; it < pre; ++it)
        tma_load_2d(stages + (size_t)it * a.stage_bytes + a.b_off, &tx, (k_begin + it) * kTcBK, m0,
                    &full[it]);
      int issued = pre;  // iterations whose copies were requested
      for (int it = pre; it < nk; ++it) {
        const int s = it % a.nstages;
        const uint32_t ph = (uint32_t)(it / a.nstages) & 1u;
        if (!mbar_wait_bounded(&empty[s], ph ^ 1u)) {
          // the stage was never released: request nothing more
          timed_out = true;
          atomicOr(&g_tc_status, SQ_DEV_TIMEOUT);
          break;
        }
        uint8_t* st = stages + (size_t)s * a.stage_bytes;
        const int k0 = (k_begin + it) * kTcBK;
        mbar_arrive_expect_tx(&full[s], bytes);
        tma_load_2d(st + wdst, &tw, wx(k0), (int)(tile * kTcBM), &full[s]);
        if (SILU) tma_load_2d(st + wdst_up, &tw, wx(k0), (int)(a.N + tile * kTcBM), &full[s]);
        tma_load_2d(st + a.b_off, &tx, k0, m0, &full[s]);
        issued = it + 1;
      }
      if (timed_out) {
        // each stage has at most one request outstanding (its last): wait for
        // it (bounded) so that no copy lands after the CTA has left
        for (int s = 0; s < a.nstages && s < issued; ++s) {
          const int last = s + ((issued - 1 - s) / a.nstages) * a.nstages;
          mbar_wait_bounded(&full[s], (uint32_t)(last / a.nstages) & 1u, 1u << 20);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // --------------------------------------------------------- MMA issuer
      for (int it = 0; it < nk; ++it) {
        const int s = it % a.nstages;
        const uint32_t ph = (uint32_t)(it / a.nstages) & 1u;
        if (!mbar_wait_bounded(QUANT ? &conv[s] : &full[s], ph)) {
          // the stage never arrived: issue no MMA on it or after it (the
          // commit below still tracks every MMA issued so far)
          timed_out = true;
          atomicOr(&g_tc_status, SQ_DEV_TIMEOUT);
          break;
        }
        tc_fence_after();
        const uint32_t st = smem_u32(stages + (size_t)s * a.stage_bytes);
        const uint64_t ad = sw128_desc(st);
        const uint64_t au = sw128_desc(st + kTcStageA);
        const uint64_t bd = sw128_desc(st + a.b_off);
#pragma unroll
        for (int kk = 0; kk < kTcBK / 16; ++kk) {
          const uint32_t acc = (it > 0 || kk > 0) ? 1u : 0u;
          // advancing 16 fp16 along K inside the swizzled row = +32 bytes
          tc_mma_f16(tmem, ad + 2 * kk, bd + 2 * kk, a.idesc, acc);
          if (SILU) tc_mma_f16(tmem + a.NB, au + 2 * kk, bd + 2 * kk, a.idesc, acc);
        }
        tc_commit(&empty[s]);
      }
      tc_commit(accf);
    }
  } else {
    // ------------------------------------- converters (quantised), epilogue
    if constexpr (QUANT) {
      if constexpr (WK == 1) {
        // INT4: this CTA's group scales (128 rows x the groups its K range
        // touches, gate and up) into shared memory once, before waiting on
        // the previous kernel: scales never depend on it, and the per-stage
        // conversion then never waits on a global load
        const int ct = tid - 64;
        const int64_t G = a.K / 128;
        const int64_t wrows = SILU ? 2 * a.N : a.N;
        const int g_lo = (k_begin * kTcBK) >> 7;
        const int ng = nk > 0 ? (((k_end * kTcBK) - 1) >> 7) + 1 - g_lo : 0;
        __half* sblk = reinterpret_cast<__half*>(smem + a.sc_off);
        for (int r = ct; r < (SILU ? 2 : 1) * kTcBM; r += 32 * EW) {
          const int h = r / kTcBM, rr = r - h * kTcBM;
          const int64_t wrow = (h ? a.N : 0) + tile * kTcBM + rr;
          const __half* src = reinterpret_cast<const __half*>(a.scales) + wrow * G + g_lo;
          __half* dst = sblk + (size_t)r * a.sc_ng;
          for (int gi = 0; gi < ng; ++gi) dst[gi] = wrow < wrows ? __ldg(src + gi) : __ushort_as_half(0);
        }
        named_bar_sync(1, 32 * EW);  // the converter warps
      }
    }
    griddep_wait();
    if constexpr (QUANT) {
      const int ct = tid - 64;  // 0 .. 32 * converter warps - 1
      const int g_lo = (k_begin * kTcBK) >> 7;
      const __half* sblk = reinterpret_cast<const __half*>(smem + a.sc_off);
      for (int it = 0; it < nk; ++it) {
        const int s = it % a.nstages;
        const uint32_t ph = (uint32_t)(it / a.nstages) & 1u;
        const int gi = (((k_begin + it) * kTcBK) >> 7) - g_lo;  // this stage's group
        if (!timed_out && !mbar_wait_bounded(&full[s], ph)) {
          timed_out = true;
          if (lane == 0) atomicOr(&g_tc_status, SQ_DEV_TIMEOUT);
        }
        uint8_t* st = stages + (size_t)s * a.stage_bytes;
#pragma unroll
        for (int h = 0; h < (SILU ? 2 : 1); ++h) {
          const uint8_t* codes = st + a.c_off + h * a.c_bytes;
          uint8_t* at = st + h * kTcStageA;
          // one job = 16 code bytes of one row: 32 INT4 / 16 FP8 weights,
          // i.e. 4 / 2 of the row's eight 16-byte fp16 chunks.  Per warp the
          // code loads cover 512 contiguous bytes and each quarter-warp's
          // chunk stores hit 8 distinct 16-byte bank groups (swizzle), so
          // neither conflicts.
          constexpr int kJobsPerRow = WK == 1 ? 2 : 4;
          constexpr int kChunksPerJob = 8 / kJobsPerRow;
#pragma unroll
          for (int job = ct; job < kTcBM * kJobsPerRow; job += 32 * EW) {
            const int row = job / kJobsPerRow, jp = job % kJobsPerRow;
            const uint4 cw = *reinterpret_cast<const uint4*>(codes + row * (kTcBK * (WK == 1 ? 1 : 2) / 2) +
                                                             jp * 16);
            uint8_t* arow = at + row * 128;
            if constexpr (WK == 2) {
              const uint32_t wv[4] = {cw.x, cw.y, cw.z, cw.w};
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                uint4 out;
                out.x = e4m3x2_to_f16x2(lo16(wv[2 * q]));
                out.y = e4m3x2_to_f16x2(hi16(wv[2 * q]));
                out.z = e4m3x2_to_f16x2(lo16(wv[2 * q + 1]));
                out.w = e4m3x2_to_f16x2(hi16(wv[2 * q + 1]));
                const int c = jp * kChunksPerJob + q;
                *reinterpret_cast<uint4*>(arow + ((c ^ (row & 7)) << 4)) = out;
              }
            } else {
              const __half2 s2 = __half2half2(sblk[(size_t)(h * kTcBM + row) * a.sc_ng + gi]);
              auto mul = [&](uint32_t v) {
                const __half2 r = __hmul2(*reinterpret_cast<const __half2*>(&v), s2);
                return *reinterpret_cast<const uint32_t*>(&r);
              };
              const uint32_t wv[4] = {cw.x, cw.y, cw.z, cw.w};
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                uint32_t v[4];
                int4x8_to_f16x2(wv[q], v);  // (k0,k4),(k1,k5),(k2,k6),(k3,k7)
                uint4 out;
                out.x = mul(__byte_perm(v[0], v[1], 0x5410));  // (k0, k1)
                out.y = mul(__byte_perm(v[2], v[3], 0x5410));  // (k2, k3)
                out.z = mul(__byte_perm(v[0], v[1], 0x7632));  // (k4, k5)
                out.w = mul(__byte_perm(v[2], v[3], 0x7632));  // (k6, k7)
                const int c = jp * kChunksPerJob + q;
                *reinterpret_cast<uint4*>(arow + ((c ^ (row & 7)) << 4)) = out;
              }
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&conv[s]);
      }
    }
  }
  if (warp >= 2) {
    // --------------------------------------------------------- epilogue
    if (!mbar_wait_bounded(accf, 0u)) {
      timed_out = true;
      if (lane == 0) atomicOr(&g_tc_status, SQ_DEV_TIMEOUT);
    }
    tc_fence_after();
  }
  if (S > 1) {
    __syncwarp();
    // every CTA of the cluster has begun, or, where partial tiles go over the
    // stages, has its MMAs behind it
    if (!a.part_off) cluster_arrive();
    cluster_wait();
  }
  const int M = CB ? min(a.NB, a.M - m0) : a.M;
  const __half* resid = CB && a.residual ? a.residual + (int64_t)m0 * a.N : a.residual;
  __half* out = CB ? a.y + (int64_t)m0 * a.N : a.y;
  const int cper = (M + S - 1) / S;  // columns of the output each rank finishes
  if (warp >= 2) {
    const int q = warp & 3;  // TMEM sub-partition this warp may read
    const int row = q * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
    const int64_t n = tile * kTcBM + row;
    // The two warps of a sub-partition share the columns in blocks of 16: every
    // other one each or, pushed without the gate from 80 columns on, the halves of
    // the row, so that they write to different ranks (FP16: unsplit 131072 x 1024
    // at 256 rows, halves 94 us, every other one 84; gate/up, N = 2048, K = 4096,
    // 64 rows 15.0 and 13.7; INT4 1.5B q/k/v, 33 rows, 6.0 and 5.6; but 7B q/k/v,
    // S = 4, at 256 rows 17.4 and 18.2).
    if (S == 1) {
      for (int c0 = warp < 6 ? 0 : 16; c0 < a.NB; c0 += 4 * EW) {
        float g[16], u[16];
        tc_ld16(taddr + (uint32_t)c0, g);
        if (SILU) tc_ld16(taddr + (uint32_t)(a.NB + c0), u);
        if (n < a.N) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int m = c0 + j;
            if (m >= M) break;
            float v = g[j];
            if constexpr (WK == 2) v *= reinterpret_cast<const float*>(a.scales)[n];
            if (a.bias) v += __half2float(a.bias[n]);
            if (SILU) {
              float uu = u[j];
              if constexpr (WK == 2) uu *= reinterpret_cast<const float*>(a.scales)[a.N + n];
              if (a.bias) uu += __half2float(a.bias[a.N + n]);
              v = v / (1.0f + expf(-v)) * uu;
            }
            if (resid) v += __half2float(resid[(int64_t)m * a.N + n]);
            out[(int64_t)m * a.N + n] = __float2half_rn(v);
          }
        }
      }
    } else {
      // Column m of the partial tile goes straight from TMEM to the rank that
      // finishes it, m / cper, at [this rank][m % cper][row]: a warp's store
      // is 32 consecutive rows, 128 bytes of one column, and nothing waits
      // for it before the barrier.  SiLU: up columns behind the gate ones.
      const int cols = a.NB * (SILU ? 2 : 1), half = (cols / 16 + 1) / 2 * 16;
      const bool halves = EW == 8 && !SILU && a.NB > 64;
      const int cend = halves && warp < 6 ? half : cols;
      for (int c0 = warp < 6 ? 0 : halves ? half : 16; c0 < cend; c0 += halves ? 16 : 4 * EW) {
        float v[16];
        tc_ld16(taddr + (uint32_t)c0, v);
        const int up = SILU && c0 >= a.NB ? 1 : 0;
        const int mb = c0 - up * a.NB;
        int owner = mb / cper, mc = mb - owner * cper;
        const int off = (((int)rank * (SILU ? 2 : 1) + up) * cper * kTcBM + row) * 4;
        const uint32_t base = smem_u32(smem) + (uint32_t)a.part_off + (uint32_t)off;
        uint32_t remote = map_rank(base, (uint32_t)min(owner, S - 1));
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (mb + j < M) st_dsmem_f32(remote + (uint32_t)(mc * kTcBM * 4), v[j]);
          if (++mc == cper) {
            mc = 0;
            ++owner;
            remote = map_rank(base, (uint32_t)min(owner, S - 1));
          }
        }
      }
    }
  }

  tc_fence_before();
  if (S > 1) {
    __syncwarp();
    cluster_sync();  // every partial column has arrived
    if (warp >= 2) {
      // This rank's columns, one element per thread and four such in flight;
      // a warp takes 32 consecutive rows.  The partials are added in rank
      // order.  Columns rather than rows per rank, and pushed rather than
      // fetched after the barrier: fetching a few rows of every column came
      // in 64-byte pieces with their latency exposed (1.5B FP16 qkv, S = 6,
      // 80 / 256 rows: 9.5 -> 6.8 / 19.8 -> 12.5 us; 7B pass at 256 rows
      // 963 -> 896; 1.5B FP8 pass at 40 rows 1320 -> 1174).
      const float* part = reinterpret_cast<const float*>(smem + a.part_off);
      const int nthr = 32 * EW;
      const int m_lo = min((int)rank * cper, M);
      const int items = (min(m_lo + cper, M) - m_lo) * kTcBM;
      const int pstep = (SILU ? 2 : 1) * cper * kTcBM;  // floats from rank to rank
      constexpr int kIt = 4;
      for (int i0 = tid - 64; i0 < items; i0 += kIt * nthr) {
        float g[kIt], u[kIt], res[kIt];
        bool live[kIt];
#pragma unroll
        for (int j = 0; j < kIt; ++j) {
          const int i = i0 + j * nthr;
          const int64_t n = tile * kTcBM + i % kTcBM;
          live[j] = i < items && n < a.N;
          g[j] = u[j] = res[j] = 0.0f;
          if (live[j] && resid)
            res[j] = __half2float(resid[(int64_t)(m_lo + i / kTcBM) * a.N + n]);
        }
        for (int qq = 0; qq < S; ++qq) {
#pragma unroll
          for (int j = 0; j < kIt; ++j) {
            const int i = i0 + j * nthr;
            if (live[j]) {
              g[j] += part[qq * pstep + i];
              if (SILU) u[j] += part[qq * pstep + cper * kTcBM + i];
            }
          }
        }
#pragma unroll
        for (int j = 0; j < kIt; ++j) {
          if (!live[j]) continue;
          const int i = i0 + j * nthr;
          const int64_t n = tile * kTcBM + i % kTcBM;
          float v = g[j];
          if constexpr (WK == 2) v *= reinterpret_cast<const float*>(a.scales)[n];
          if (a.bias) v += __half2float(a.bias[n]);
          if (SILU) {
            float uu = u[j];
            if constexpr (WK == 2) uu *= reinterpret_cast<const float*>(a.scales)[a.N + n];
            if (a.bias) uu += __half2float(a.bias[a.N + n]);
            v = v / (1.0f + expf(-v)) * uu;
          }
          if (resid) v += res[j];
          out[(int64_t)(m_lo + i / kTcBM) * a.N + n] = __float2half_rn(v);
        }
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(a.tmem_cols)
                 : "memory");
  }
}

// ---------------------------------------------------------------- host side

static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// [rows, inner] row-major -> 2-D tensor map with box (box_inner, box_rows);
// zero fill outside the tensor.
static bool make_map(CUtensorMap* m, const void* base, CUtensorMapDataType dt, int elem_bytes,
                     int64_t rows, int64_t inner, int box_inner, int box_rows,
                     CUtensorMapSwizzle swz) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)inner * (cuuint64_t)elem_bytes};
  cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// instruction descriptor, kind::f16: D fp32, A and B fp16, both K-major,
// N = nb, M = 128
static uint32_t make_idesc(int nb) {
  uint32_t d = 0;
  d |= 1u << 4;                       // D format fp32
  d |= (uint32_t)(nb >> 3) << 17;     // N / 8
  d |= (uint32_t)(kTcBM >> 4) << 24;  // M / 16
  return d;
}

bool tc_supported(int M, int64_t K, int epi) {
  (void)epi;
  return M >= 1 && M <= 256 && K % 8 == 0 && tensor_map_encoder() != nullptr;
}

// Raises the kernel's dynamic shared-memory limit to `smem` (once per size
// and device) and allows cluster sizes above 8.
template <int WK, bool SILU, bool CB, int EW>
static cudaError_t tc_prepare(size_t smem) {
  auto k = tc_linear_kernel<WK, SILU, CB, EW>;
  static int smem_set[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if ((int)smem > smem_set[dev]) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    smem_set[dev] = (int)smem;
  }
  return cudaSuccess;
}

// Clusters of S CTAs (with `smem` bytes each) that can be resident at once,
// from the occupancy calculator; cached per device, S and size.
template <int WK, bool SILU, bool CB, int EW>
static int tc_max_clusters(int S, size_t smem) {
  struct Entry {
    size_t smem;
    int n;
  };
  static Entry cache[64][kTcMaxSplit + 1][4] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || S < 1 || S > kTcMaxSplit) return 0;
  for (Entry& en : cache[dev][S])
    if (en.smem == smem + 1) return en.n;
  if (tc_prepare<WK, SILU, CB, EW>(smem) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)S, 1, 1);
  cfg.blockDim = dim3(tc_threads(EW));
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, tc_linear_kernel<WK, SILU, CB, EW>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  for (Entry& en : cache[dev][S])
    if (en.smem == 0) {
      en.smem = smem + 1;
      en.n = n;
      break;
    }
  return n;
}

// Clusters of S CTAs that a split may take with two CTAs per SM, 152 SMs: as many
// as run at once, measured at K = 8192 by the tile count at which a second wave
// begins (74, 58 of four, five CTAs; 14 of 14 to 16; of 13 three more run, but
// twelve CTAs are faster), and above five CTAs at most 5/6 of the places.  Up to
// 46 of six, 38 of seven, 30 of nine, 28 of ten run alone, but behind another
// kernel, whose last CTAs still hold places, some wait: 7B FP16 at three rows, 28
// tiles, S = 9 / 10, four layers without lm_head 332 / 367 us.
static const int kTcClusters[kTcMaxSplit + 1] = {0, 304, 152, 101, 74, 58, 42, 36, 31, 28, 25, 22, 21, 16, 14, 14, 14};

// Split-K factor.  FP16 and FP8 weights (HBM-bound): double S while the
// split tiles still fill at most half the SMs, so that the next kernel's
// CTAs find free SMs and start their weight loads early (programmatic
// dependent launch) -- filling every SM measured slower on the 7B shapes.
// INT4 weights (bound by the in-CTA dequantisation): the S in
// 1..kTcMaxSplit that minimises (waves of resident clusters) x (k-steps per
// CTA + 2 for the split reduction), at least 2 k-steps per CTA; ties keep
// the smaller S.
template <int WK, bool SILU, bool CB, int EW>
static int tc_pick_split(int64_t tiles, int ksteps, size_t smem, int max_split, bool two_per_sm,
                         bool int4_large, int many_rows_steps) {
  if (WK == 1 && int4_large) {
    // two CTAs per SM: the largest power-of-two split with at most 2.2 CTAs
    // per SM in all and at least 12 k-steps per CTA (odd splits of 3 and 7
    // measured 20-50 % slower than their neighbours)
    const int sms = device_sm_count();
    int S = 1;
    for (int s = 2; s <= max_split && s <= kTcMaxSplitInt4; s <<= 1)
      if (tiles * s * 10 <= 22 * (int64_t)sms && ksteps >= 12 * s) S = s;
    return S;
  }
  if (WK != 1) {
    const int sms = device_sm_count();
    int S = 1;
    if (two_per_sm) {
      // two CTAs per SM: the largest S (up to 16) whose clusters all run at once
      // (1.5B down projection, M = 5: 10.4 -> 8.7 us from S = 8 to 16).  Clusters
      // leave places of a GPC unused, so fewer run than there are places for
      // (kTcClusters).  One too many costs a second wave: FP16 gate/up, K = 8192, 8 rows, 14 / 15 tiles at S = 16
      // 13.7 / 21.4 us, 16 / 17 at S = 13 15.0 / 16.3 (no wave, but 15.8 at S =
      // 12), 58 / 59 at S = 5 45.2 / 57.2.
      while (S < max_split && ksteps >= 4 * (S + 1) &&
             tiles * kNumSMs <= kTcClusters[S + 1] * (int64_t)sms)
        ++S;
      return S;
    }
    // one CTA per SM: clusters of at most the portable 8 SMs
    if (many_rows_steps > 0) {
      // many activation rows (NB > 64: every k-step also streams a large
      // activation tile and runs a long MMA): the largest S that still fits
      // one wave, with many_rows_steps k-steps per CTA (six with column blocks:
      // 1.5B o at 256 rows S = 4 8.7 us, S = 5 8.9)
      while (S + 1 <= max_split && S + 1 <= 8 && tiles * (S + 1) <= sms && ksteps >= many_rows_steps * (S + 1))
        ++S;
      return S;
    }
    while (2 * S <= max_split && 2 * S <= 8 && tiles * S * 2 <= sms && ksteps >= 4 * S * 2) S <<= 1;
    return S;
  }
  int best_s = 1;
  int64_t best = INT64_MAX;
  for (int S = 1; S <= max_split && S <= kTcMaxSplitInt4 && ksteps >= 2 * S; ++S) {
    const int nc = tc_max_clusters<WK, SILU, CB, EW>(S, smem);
    if (nc <= 0) continue;
    const int64_t waves = (tiles + nc - 1) / nc;
    const int64_t cost = waves * ((ksteps + S - 1) / S + (S > 1 ? 2 : 0));
    if (cost < best) {
      best = cost;
      best_s = S;
    }
  }
  return best_s;
}

// Shared memory of ns stages: the stages, the barriers, the INT4 scale block.
static int tc_sc_off(const TcArgs& a, int ns) { return (ns * a.stage_bytes + (3 * ns + 2) * 8 + 16 + 15) / 16 * 16; }
static size_t tc_smem(const TcArgs& a, int ns) { return 1024 + (size_t)tc_sc_off(a, ns) + (size_t)a.sc_bytes; }
// ... and a partial tile of `part` bytes behind them.
static size_t tc_part_end(const TcArgs& a, int ns, size_t part) { return (tc_smem(a, ns) + 127) / 128 * 128 + part; }

template <int WK, bool SILU, bool CB, int EW>
static cudaError_t tc_launch_inst(const CUtensorMap& tw, const CUtensorMap& tx, TcArgs a,
                                  int64_t tiles, size_t smem, cudaStream_t st) {
  auto k = tc_linear_kernel<WK, SILU, CB, EW>;
  cudaError_t e = tc_prepare<WK, SILU, CB, EW>(smem);
  if (e != cudaSuccess) return e;
  const int S = tc_pick_split<WK, SILU, CB, EW>(tiles * a.colblocks, a.ksteps, smem, a.max_split, a.two_per_sm != 0,
                                       a.int4_large != 0, a.colblocks > 1 ? 6 : a.NB > 64 ? 4 : 0);
  a.splits = S;
  // The partial tile beside the stages where that costs no residency, and then no
  // more stages than a CTA has k-steps: the ranks push without waiting for each
  // other's MMAs, and one of the two cluster barriers between the last MMA and the
  // output, about half a microsecond, is long past (FP16 896 x 4864, 9 rows: 5.3 ->
  // 4.6 us; 1.5B q/k/v, 16 rows: 5.2 -> 4.3).  Up to 16 rows four stages rather than
  // five keep two CTAs within 2 x 97 KB: above that the SM's shared-memory
  // configuration differs from that of the kernels around, which start later (28
  // layers of 1.5B at 9 rows 807 us without that, 774 with; a 1.5B decoder pass of
  // five tokens 1474 and 1456; at 24 rows 97 KB as a bound for all 882, so 852).
  a.part_off = 0;
  if (S > 1) {
    const int nk = (a.ksteps + S - 1) / S;
    int ns = a.nstages < nk ? a.nstages : nk < 2 ? 2 : nk;
    const size_t part = (size_t)S * (((a.M < a.NB ? a.M : a.NB) + S - 1) / S) * (SILU ? 2 : 1) * kTcBM * 4;
    const size_t limit = (size_t)(!a.two_per_sm ? 227 : a.NB > 16 ? 113 : 97) * 1024;
    while (a.two_per_sm && a.NB == 16 && ns > 4 && tc_part_end(a, ns, part) > limit) --ns;
    if (tc_part_end(a, ns, part) <= limit) {
      a.nstages = ns;
      a.sc_off = tc_sc_off(a, ns);
      smem = tc_part_end(a, ns, part);
      a.part_off = (int)(smem - part - 1024);
      e = tc_prepare<WK, SILU, CB, EW>(smem);
      if (e != cudaSuccess) return e;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)S, (unsigned)tiles, (unsigned)a.colblocks);
  cfg.blockDim = dim3(tc_threads(EW));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int na = 0;
  attr[na].id = cudaLaunchAttributeClusterDimension;
  attr[na].val.clusterDim.x = (unsigned)S;
  attr[na].val.clusterDim.y = 1;
  attr[na].val.clusterDim.z = 1;
  ++na;
  const bool legacy = (st == nullptr || st == cudaStreamLegacy || st == cudaStreamPerThread);
  if (!legacy && pdl_enabled()) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, k, tw, tx, a);
}

cudaError_t launch_tc(int wk, const __half* x, const void* w, const void* scales, const __half* bias,
                      const __half* residual, __half* y, int M, int64_t N, int64_t K, int epi,
                      cudaStream_t st) {
  const bool silu = epi == SQ_EPI_SILU_GATE;
  const int64_t tiles = (N + kTcBM - 1) / kTcBM;
  const int sms = device_sm_count();
  // Short rows (K <= 2048) under many activation rows: the tail after the last
  // MMA costs more than the products, and the few tiles leave SMs idle, so two
  // CTAs take half of the activation rows each where they fit beside each other.
  // FP16 (a quantised tile would be converted twice), 1.5B, one block -> two:
  // at 144 / 256 rows gate/up 21.4 -> 19.1 / 29.5 -> 21.3 us, q/k/v 8.4 -> 7.8 /
  // 12.2 -> 9.3, o 7.9 -> 7.1 / 12.0 -> 8.7; at 80 rows the gate/up loses (16.8
  // against 17.5), and so do longer rows (7B q/k/v at 256 rows 17.5 against 18.8).
  const int colblocks = wk == SQ_W_FP16 && M > 96 && K <= 2048 && 2 * tiles <= sms ? 2 : 1;
  const int nb = ((M + colblocks - 1) / colblocks + 15) / 16 * 16;
  const int64_t wrows = silu ? 2 * N : N;
  CUtensorMap tw, tx;
  bool ok;
  int c_bytes = 0;
  if (wk == SQ_W_FP16) {
    ok = make_map(&tw, w, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, wrows, K, kTcBK, kTcBM,
                  CU_TENSOR_MAP_SWIZZLE_128B);
  } else if (wk == SQ_W_FP8) {
    c_bytes = kTcBM * kTcBK;  // 64 codes per row
    ok = make_map(&tw, w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, wrows, K, kTcBK, kTcBM,
                  CU_TENSOR_MAP_SWIZZLE_NONE);
  } else {
    c_bytes = kTcBM * kTcBK / 2;  // 64 nibbles = 32 bytes per row
    ok = make_map(&tw, w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, wrows, K / 2, kTcBK / 2, kTcBM,
                  CU_TENSOR_MAP_SWIZZLE_NONE);
  }
  ok = ok && make_map(&tx, x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, M, K, kTcBK, nb,
                      CU_TENSOR_MAP_SWIZZLE_128B);
  if (!ok) return cudaErrorInvalidValue;
  TcArgs a = {};
  a.scales = scales;
  a.M = M;
  a.NB = nb;
  a.colblocks = colblocks;
  a.N = N;
  a.K = K;
  a.epi = epi;
  a.ksteps = (int)((K + kTcBK - 1) / kTcBK);
  a.bias = bias;
  a.residual = residual;
  a.y = y;
  a.idesc = make_idesc(nb);
  const int S2 = silu ? 2 : 1;
  const int cols = nb * S2;
  int tc = 32;
  while (tc < cols) tc <<= 1;
  a.tmem_cols = tc;
  const int a_bytes = kTcStageA * S2;
  const int b_bytes = (nb * 128 + 1023) / 1024 * 1024;
  a.b_off = a_bytes;
  a.c_off = a_bytes + b_bytes;
  a.c_bytes = c_bytes;
  a.stage_bytes = a.c_off + (c_bytes * S2 + 1023) / 1024 * 1024;
  // the split of K over a cluster is chosen per kernel instance (occupancy)
  // INT4: room for a CTA's group scales, sized for an unsplit K range
  // (a range of n stages touches at most (n - 1) / 2 + 2 groups)
  a.sc_ng = 0;
  size_t sc_bytes = 0;
  if (wk == SQ_W_INT4) {
    const int64_t G = K / 128;
    const int64_t need = (a.ksteps - 1) / 2 + 2;
    a.sc_ng = (int)(need < G ? need : G);
    sc_bytes = (size_t)S2 * kTcBM * (size_t)a.sc_ng * 2;
  }
  // Few activation rows (NB <= 64) and few row tiles: stages for two CTAs per
  // SM (100 KB each) and a deeper split, so every SM streams and one
  // CTA's prologue and epilogue overlap the other's loads (measured 8-28 %
  // faster on the 1.5B/7B down, qkv and o shapes); otherwise one CTA per SM
  // with 200 KB of stages.
  // INT4 weights of 20 MB and more at NB <= 64 (the draft pass at 8 or 16
  // rows: 7B/14B gate/up, down and lm_head) take two CTAs per SM too, with a
  // power-of-two split: measured 20-40 % faster than one CTA per SM with the
  // occupancy cost model (14B lm_head at M = 16: 332 -> 203 us; gate/up 57
  // -> 45 us; down 45 -> 36 us).
  const double wbytes = (double)wrows * (double)(K / 2) + (double)wrows * (double)(K / 128) * 2.0;
  a.int4_large = (wk == SQ_W_INT4 && nb <= 64 && wbytes >= 20e6) ? 1 : 0;
  // FP16 without the gate and from 24 tiles on: also up to 96 rows, and up to
  // 128 from 40 tiles on (one CTA per SM -> two: 14B q/k/v, o, down at 80 rows
  // 21.7, 16.8, 34.1 -> 17.2, 14.5, 29.8 us, at 112 rows 22.9, 17.6, 35.1 ->
  // 19.1, 16.4, 32.1; four 7B layers at 80 rows 456 -> 389, but its 28 and 36
  // tiles at 112 rows 12.9, 11.9 against 13.5, 12.2; 1.5B, 12 and 16 tiles, 28
  // layers at 80 rows 1153 against 1184; 14B FP8 at 80 rows 518 against 535).
  const bool more_rows =
      wk == SQ_W_FP16 && !silu && colblocks == 1 && tiles >= 24 && (nb <= 96 || (nb <= 128 && tiles >= 40));
  a.two_per_sm = (a.int4_large || (tiles * 2 <= sms && ((nb <= 64 && colblocks == 1) || more_rows))) ? 1 : 0;
  const int budget = (a.two_per_sm ? 100 : 200) * 1024;
  int ns = (int)((budget - (int64_t)sc_bytes) / a.stage_bytes);
  if (ns > 8) ns = 8;
  if (ns < 2) ns = 2;
  a.nstages = ns;
  // split-K: a rank gathers the fp32 partials of its ceil(M / S) columns from
  // all S ranks in the (then idle) stage memory; the split stays where they fit
  a.max_split = 1;
  while (a.max_split < kTcMaxSplit) {
    const int s1 = a.max_split + 1;
    if ((size_t)s1 * (((M < nb ? M : nb) + s1 - 1) / s1) * S2 * kTcBM * 4 > (size_t)ns * a.stage_bytes) break;
    ++a.max_split;
  }
  a.sc_bytes = (int)sc_bytes;
  a.sc_off = tc_sc_off(a, ns);
  const size_t smem = tc_smem(a, ns);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  if (colblocks > 1)
    return silu ? tc_launch_inst<SQ_W_FP16, true, true, 8>(tw, tx, a, tiles, smem, st)
                : tc_launch_inst<SQ_W_FP16, false, true, 8>(tw, tx, a, tiles, smem, st);
  if (wk == SQ_W_FP16 && nb == 16)
    return silu ? tc_launch_inst<SQ_W_FP16, true, false, 4>(tw, tx, a, tiles, smem, st)
                : tc_launch_inst<SQ_W_FP16, false, false, 4>(tw, tx, a, tiles, smem, st);
#define SQ_TC_CASE(WK_)                                                                \
  if (wk == WK_) return silu ? tc_launch_inst<WK_, true, false, 8>(tw, tx, a, tiles, smem, st)  \
                             : tc_launch_inst<WK_, false, false, 8>(tw, tx, a, tiles, smem, st);
  SQ_TC_CASE(SQ_W_FP16)
  SQ_TC_CASE(SQ_W_INT4)
  SQ_TC_CASE(SQ_W_FP8)
#undef SQ_TC_CASE
  return cudaErrorInvalidValue;
}

// Failure-path self-test: one thread waits, with the tile kernel's bounded
// poll loop, on an mbarrier that nothing arrives at; after `polls` polls it
// gives up and sets SQ_DEV_TIMEOUT, exactly as a tile kernel's wait would.
// Nothing is in flight (no bulk copy, no MMA), so giving up is clean.
__global__ void wait_selftest_poll_kernel(uint32_t polls) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait_bounded(&bar, 0, polls)) atomicOr(&g_tc_status, SQ_DEV_TIMEOUT);
}

cudaError_t launch_wait_selftest_poll(uint32_t polls, cudaStream_t st) {
  wait_selftest_poll_kernel<<<1, 32, 0, st>>>(polls);
  return cudaGetLastError();
}

cudaError_t take_tc_status(uint32_t* bits) {
  uint32_t v = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_tc_status, sizeof(v));
  if (e != cudaSuccess) return e;
  if (v) e = cudaMemcpyToSymbol(g_tc_status, &zero, sizeof(zero));
  *bits |= v;
  return e;
}

}  // namespace sq
