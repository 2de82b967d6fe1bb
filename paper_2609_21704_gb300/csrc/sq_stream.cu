// sq_stream.cu -- linear layer for up to sixteen activation rows (the draft
// pass, Sec. III-D.2; the verify pass of one or two sequences, Sec. III-D.3):
// weights streamed once from memory, products on the tensor cores'
// register-operand path (mma.sync m16n8k16, fp16 inputs, fp32 sums).
//
// Work split: every CTA (or cluster of KS CTAs along K) owns an equal
// contiguous share of the output ROWS, cut into tiles of at most sixteen
// rows of equal height: tiles are padded, memory traffic is not, so no SM
// reads a row more than another (whole 16-row tiles left a third of the SMs
// idle at 320 tiles).  Inside a CTA the warps take (tile, part of K) jobs; the
// parts meet in shared memory and are added in a fixed order.
//
// Stream: a lane copies the 16-byte pieces that it multiplies itself into its
// own slots of a shared-memory ring (cp.async, no barrier between lanes),
// the first ones before the wait on the kernel that produces x.  Up to eight
// rows a CTA keeps to 80 registers a thread and, where it has little to
// stream, to half the shared memory: the next launch's CTA fits beside it and
// its first copies run while this one computes.  A call with much to stream
// takes more than half, so that none does.
//
// Products: A = sixteen weight rows, B = the activation rows as columns (eight
// a tile; columns past M repeat a row and are dropped).  FP16 pieces are
// operands as they are, E4M3 codes are converted (exactly), INT4 nibbles to the
// exact integers c, nine instructions for eight weights, four of them fp16
// arithmetic.  Masked nibbles as fp16 subnormals, their offset removed per group
// of 128, take five, but a product with a subnormal keeps seven bits fewer beside
// the others of its sum (gated activations: 4 % of the fp16 results wrongly
// rounded against 0.06 %), and the offset's sums cost more than the four: 14B at
// 16 rows, four layers and lm_head, 451 us against 426, 1.5B at 8 rows 804
// against 732; only one row loses (14B lm_head 4 to 6 us).
#include <mutex>

#include "sq_internal.h"
#include "sq_stream_plan.h"

namespace sq {

namespace {

struct SArgs : StreamPlan {
  const __half* x;         // [M, K]
  const uint8_t* w;        // weight rows
  const void* scales;      // INT4 fp16 [rows, K/128]; FP8 fp32 [rows]
  const __half* bias;
  const __half* residual;
  __half* y;
  const __half* gamma;     // RMSNorm gains or null: x is normalised while staged
  float eps;
};

__device__ __forceinline__ void s_mma(float d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                      uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same from zero
__device__ __forceinline__ void s_mma0(float d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                       uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.0f));
}
__device__ __forceinline__ uint4 s_lds16(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr));
  return v;
}
__device__ __forceinline__ float s_ld_rank(const float* local, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
  return v;
}
__device__ __forceinline__ void s_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void s_cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// RMSNorm of two fp16 values as the standalone kernel rounds them.
__device__ __forceinline__ uint32_t s_norm2(uint32_t xw, uint32_t gw, float r) {
  const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&xw));
  const float2 g = __half22float2(*reinterpret_cast<const __half2*>(&gw));
  const __half2 h = __floats2half2_rn(__fmul_rn(__fmul_rn(x.x, r), g.x), __fmul_rn(__fmul_rn(x.y, r), g.y));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// y[m, n] from the fp32 dot product v (and the up row's u).
template <int WK, bool SILU>
__device__ __forceinline__ void s_store(const SArgs& a, int64_t n, int m, float v, float u) {
  if constexpr (WK == SQ_W_FP8) v *= reinterpret_cast<const float*>(a.scales)[n];
  if (a.bias) v += __half2float(a.bias[n]);
  if constexpr (SILU) {
    if constexpr (WK == SQ_W_FP8) u *= reinterpret_cast<const float*>(a.scales)[a.N + n];
    if (a.bias) u += __half2float(a.bias[a.N + n]);
    v = v / (1.0f + expf(-v)) * u;
  }
  if (a.residual) v += __half2float(a.residual[(int64_t)m * a.N + n]);
  a.y[(int64_t)m * a.N + n] = __float2half_rn(v);
}

// WK: weight format; NT as above.
template <int WK, bool SILU, int NT>
__global__ void __launch_bounds__(32 * s_warps(NT), NT == 1 ? 2 : 1) stream_linear_kernel(const __grid_constant__ SArgs a) {
  constexpr int NW = s_warps(NT), NTHR = 32 * NW;
  constexpr int KU = WK == SQ_W_INT4 ? 128 : WK == SQ_W_FP8 ? 64 : 32;  // weights of a unit
  constexpr int XU = 2 * KU;                                            // staged bytes of a unit
  constexpr int WR = SILU ? 2 : 1;                                      // weight tiles of an output tile
  constexpr int US = SILU ? 1 : 2;                                      // units of a step
  constexpr int NC = NT == 2 ? 2 : 1;                                   // column tiles
  constexpr int NE = NT == 0 ? 2 : 4;                                   // sums of a lane, tile and column tile
  constexpr bool I4 = WK == SQ_W_INT4;
  extern __shared__ __align__(128) uint8_t ssm[];
  const uint32_t sbase = smem_u32(ssm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int M = NT == 0 ? 1 : a.M;
  float* rinv = reinterpret_cast<float*>(ssm + a.off_misc);
  float* nred = rinv + kMaxRows;  // [row][8]
  float* red = reinterpret_cast<float*>(ssm + a.off_red);

  const int ncl = (int)gridDim.x / a.KS;
  const int cl = (int)blockIdx.x / a.KS, rank = (int)blockIdx.x - cl * a.KS;
  const int64_t n0 = (int64_t)cl * a.N / ncl;
  const int rows = (int)((int64_t)(cl + 1) * a.N / ncl - n0);
  const int ntiles = (rows + 15) / 16;
  const int th = ntiles > 0 ? (rows + ntiles - 1) / ntiles : 1;  // rows of a tile
  const int ub = rank * a.U / a.KS;
  const int nu = (rank + 1) * a.U / a.KS - ub;  // this CTA's units
  const bool direct = a.S == 1 && a.KS == 1;

  // ---- issue side: this warp's jobs as one sequence of steps
  const uint32_t ring = sbase + a.off_ring + (uint32_t)(warp * a.ns * kSlotBytes + lane * 16);
  const int64_t rb8 = 8 * a.row_bytes;
  const int64_t upoff = a.N * a.row_bytes;
  const uint8_t* ip = nullptr;  // row g, this lane's piece, next unit
  int it0 = 0, ijj = warp, ileft = 0, inr = 0;
  auto issue_job = [&]() {
    ileft = 0;
    while (it0 < ntiles) {
      if (ijj < min(a.pass_tiles, ntiles - it0) * a.S) {
        const int tl = ijj / a.S, part = ijj - tl * a.S;
        const int row = (it0 + tl) * th, u0 = part * nu / a.S;
        inr = min(th, rows - row);
        ileft = (part + 1) * nu / a.S - u0;
        ip = a.w + (n0 + row + g) * a.row_bytes + (int64_t)(ub + u0) * 64 + t * 16;
        if (I4 && t < 2 * WR && g + 8 * (t & 1) < inr) {
          const int64_t r = (t > 1 ? a.N : 0) + n0 + row + g + 8 * (t & 1);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint16_t*>(a.scales) + r * a.U + ub + u0));
        }
        return;
      }
      it0 += a.pass_tiles;
      ijj = warp;
    }
  };
  auto issue = [&](int slot) {
    if (ileft > 0) {
      const uint32_t dst = ring + slot * kSlotBytes;
      const bool v0 = g < inr, v8 = g + 8 < inr;
      const uint8_t* q = SILU ? ip + upoff : ip + 64;
      const bool two = SILU || ileft > 1;
      if (v0) {
        s_cp16(dst, ip);
        if (two) s_cp16(dst + 1024, q);
      }
      if (v8) {
        s_cp16(dst + 512, ip + rb8);
        if (two) s_cp16(dst + 1536, q + rb8);
      }
      ip += US * 64;
      ileft -= US;
      if (ileft <= 0) {
        ijj += NW;
        issue_job();
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  issue_job();
  for (int i = 0; i < a.ns - 1; ++i) issue(i);

  // INT4 group scales of a step, fetched one step ahead: [unit or tile][row g, row g + 8]
  const uint16_t* sp = nullptr;
  const int64_t sp8 = 8 * (int64_t)a.U, spup = a.N * a.U;
  uint16_t sn[2][2];
  auto fetch = [&](bool v0, bool v8, bool two) {
    if constexpr (I4) {
      const uint16_t* q = SILU ? sp + spup : sp + 1;
      sn[0][0] = v0 ? __ldg(sp) : (uint16_t)0;
      sn[0][1] = v8 ? __ldg(sp + sp8) : (uint16_t)0;
      sn[1][0] = v0 && two ? __ldg(q) : (uint16_t)0;
      sn[1][1] = v8 && two ? __ldg(q + sp8) : (uint16_t)0;
    }
  };
  auto first_scales = [&](int row, int nr, int u0, int u1) {
    if constexpr (I4) {
      sp = reinterpret_cast<const uint16_t*>(a.scales) + (n0 + row + g) * a.U + ub + u0;
      fetch(g < nr, g + 8 < nr, SILU || u0 + 1 < u1);
    }
  };
  if (warp < min(a.pass_tiles, ntiles) * a.S) {  // the first job's, before the wait
    const int tl = warp / a.S, part = warp - tl * a.S;
    first_scales(tl * th, min(th, rows - tl * th), part * nu / a.S, (part + 1) * nu / a.S);
  }
  griddep_wait();
  griddep_launch_dependents();

  // ---- RMSNorm statistics in the standalone kernel's order: thread t takes
  // the 8-value chunks t, t + 256, ..., then warp sums, then the eight warp
  // sums in order
  if (a.gamma != nullptr) {
    if (warp < 8)
      for (int m = 0; m < M; ++m) {
        float ss = 0.0f;
        for (int c = tid; c < a.K / 8; c += 256)
          ss = sumsq8(reinterpret_cast<const uint4*>(a.x + (int64_t)m * a.K)[c], ss);
        ss = warp_sum(ss);
        if (lane == 0) nred[m * 8 + warp] = ss;
      }
    __syncthreads();
    if (tid < M) {
      float tot = 0.0f;
      for (int w = 0; w < 8; ++w) tot += nred[tid * 8 + w];
      rinv[tid] = 1.0f / sqrtf(tot / (float)a.K + a.eps);
    }
    __syncthreads();
  }

  // ---- stage x in the order of the products' operands
  {
    const int cpr = nu * (KU / 8);  // 16-byte chunks of a row
    const int total = M * cpr;
    constexpr int B = NT == 0 ? 2 : 4;
    for (int i0 = tid; i0 < total; i0 += NTHR * B) {
      uint4 v[B];
      int mm[B], cc[B];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int i = i0 + b * NTHR;
        mm[b] = NT == 0 ? 0 : i / cpr;
        cc[b] = i - mm[b] * cpr;
        if (i < total) v[b] = *reinterpret_cast<const uint4*>(a.x + (int64_t)mm[b] * a.K + ub * KU + 8 * cc[b]);
      }
#pragma unroll
      for (int b = 0; b < B; ++b) {
        if (i0 + b * NTHR >= total) break;  // (the threads of a unit break together)
        const int m = mm[b], c = cc[b];
        uint4 q = v[b];
        if (a.gamma != nullptr) {
          const uint4 gm = *reinterpret_cast<const uint4*>(a.gamma + ub * KU + 8 * c);
          const float r = rinv[m];
          q = make_uint4(s_norm2(q.x, gm.x, r), s_norm2(q.y, gm.y, r), s_norm2(q.z, gm.z, r), s_norm2(q.w, gm.w, r));
        }
        const int u = c / (KU / 8), ci = c % (KU / 8);
        uint4* dst = reinterpret_cast<uint4*>(ssm + m * a.xstride + u * XU);
        if constexpr (I4) {
          // lane t reads k = 32 t + 8 i + (0,4)(2,6)(1,5)(3,7) at [i][t]
          dst[(ci & 3) * 4 + (ci >> 2)] =
              make_uint4(__byte_perm(q.x, q.z, 0x5410), __byte_perm(q.y, q.w, 0x5410),
                         __byte_perm(q.x, q.z, 0x7632), __byte_perm(q.y, q.w, 0x7632));
        } else if constexpr (WK == SQ_W_FP8) {
          dst[(ci & 1) * 4 + (ci >> 1)] = q;  // lane t: k = 16 t + 8 i .. at [i][t]
        } else {
          dst[ci] = q;  // lane t: k = 8 t ..
        }
      }
    }
  }
  __syncthreads();

  uint32_t xa[NC];  // this lane's activation row (column g of tile i), its chunk t
#pragma unroll
  for (int i = 0; i < NC; ++i) xa[i] = sbase + (uint32_t)(min(8 * i + g, M - 1) * a.xstride + t * 16);

  // products of one 64-byte unit of a tile, every other one in d[i][0] and in
  // d[i][1]; from zero when I4
  auto unit = [&](const uint4 w0, const uint4 w1, int u, float (&d)[NC][2][4]) {
    const uint32_t r0[4] = {w0.x, w0.y, w0.z, w0.w}, r1[4] = {w1.x, w1.y, w1.z, w1.w};
    if constexpr (I4) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t p0[4], p1[4];
        int4x8_to_f16x2(r0[q], p0);
        int4x8_to_f16x2(r1[q], p1);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          const uint4 b = s_lds16(xa[i] + u * XU + q * 64);
          if (q == 0) {
            s_mma0(d[i][0], p0[0], p1[0], p0[2], p1[2], b.x, b.y);
            s_mma0(d[i][1], p0[1], p1[1], p0[3], p1[3], b.z, b.w);
          } else {
            s_mma(d[i][0], p0[0], p1[0], p0[2], p1[2], b.x, b.y);
            s_mma(d[i][1], p0[1], p1[1], p0[3], p1[3], b.z, b.w);
          }
        }
      }
    } else if constexpr (WK == SQ_W_FP8) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint4 b[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) b[i] = s_lds16(xa[i] + u * XU + h * 64);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const uint32_t c0 = r0[2 * h + p], c1 = r1[2 * h + p];
          const uint32_t a0 = e4m3x2_to_f16x2(lo16(c0)), a2 = e4m3x2_to_f16x2(hi16(c0));
          const uint32_t a1 = e4m3x2_to_f16x2(lo16(c1)), a3 = e4m3x2_to_f16x2(hi16(c1));
#pragma unroll
          for (int i = 0; i < NC; ++i) s_mma(d[i][p], a0, a1, a2, a3, p ? b[i].z : b[i].x, p ? b[i].w : b[i].y);
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        const uint4 b = s_lds16(xa[i] + u * XU);
        s_mma(d[i][0], r0[0], r1[0], r0[1], r1[1], b.x, b.y);
        s_mma(d[i][1], r0[2], r1[2], r0[3], r1[3], b.z, b.w);
      }
    }
  };

  // acc[h][i][e]: weight tile h, column tile i.  One row (NT == 0): e the rows
  // g and g + 8, column 0 (lane t = 0).  Else rows g (e < 2) and g + 8,
  // activation rows 8 i + 2 t + (e & 1).
  int slot = 0;
  bool first = true;
  for (int t0 = 0; t0 < ntiles; t0 += a.pass_tiles) {
    const int nt = min(a.pass_tiles, ntiles - t0);
    float* buf = red + ((t0 / a.pass_tiles) & 1) * a.red_floats;
    for (int jj = warp; jj < nt * a.S; jj += NW) {
      const int tl = jj / a.S, part = jj - tl * a.S;
      const int row = (t0 + tl) * th, nr = min(th, rows - row);
      const int u0 = part * nu / a.S, u1 = (part + 1) * nu / a.S;
      const bool v0 = g < nr, v8 = g + 8 < nr;
      float acc[WR][NC][NE];
#pragma unroll
      for (int h = 0; h < WR; ++h)
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
          for (int e = 0; e < NE; ++e) acc[h][i][e] = 0.0f;
      float d[WR][NC][2][4];
      if constexpr (!I4) {
#pragma unroll
        for (int h = 0; h < WR; ++h)
#pragma unroll
          for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int p = 0; p < 2; ++p) d[h][i][p][0] = d[h][i][p][1] = d[h][i][p][2] = d[h][i][p][3] = 0.0f;
      }
      if (!first) first_scales(row, nr, u0, u1);
      first = false;
      // one unit (or tile) p of a step from the slot at src
      auto part_of_step = [&](uint32_t src, int p, int uu, const uint16_t (&sc)[2]) {
        const int h = SILU ? p : 0;
        const uint4 wa = s_lds16(src + p * 1024), wb = s_lds16(src + p * 1024 + 512);
        if constexpr (I4) {
          float e[NC][2][4];
          unit(wa, wb, uu, e);
          const float s0 = __half2float(__ushort_as_half(sc[0])), s1 = __half2float(__ushort_as_half(sc[1]));
#pragma unroll
          for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int x = 0; x < NE; ++x) {
              const int q = NT == 0 ? 2 * x : x;
              acc[h][i][x] = fmaf(q < 2 ? s0 : s1, e[i][0][q] + e[i][1][q], acc[h][i][x]);
            }
        } else {
          unit(wa, wb, uu, d[h]);
        }
      };
      for (int u = u0; u < u1; u += US) {
        const bool two = SILU || u + 1 < u1;
        const uint16_t s0[2] = {sn[0][0], sn[0][1]}, s1[2] = {sn[1][0], sn[1][1]};
        if constexpr (I4) {
          if (u + US < u1) {  // the next step's
            sp += US;
            fetch(v0, v8, SILU || u + US + 1 < u1);
          }
        }
        if (a.ns == 3) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 2;" ::: "memory");
        issue(slot == 0 ? a.ns - 1 : slot - 1);
        const uint32_t src = ring + slot * kSlotBytes;
        slot = slot + 1 == a.ns ? 0 : slot + 1;
        if (two) {
          part_of_step(src, 0, u, s0);
          part_of_step(src, 1, SILU ? u : u + 1, s1);
        } else {
          part_of_step(src, 0, u, s0);
        }
      }
      if constexpr (!I4) {
#pragma unroll
        for (int h = 0; h < WR; ++h)
#pragma unroll
          for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int e = 0; e < NE; ++e) {
              const int q = NT == 0 ? 2 * e : e;
              acc[h][i][e] = d[h][i][0][q] + d[h][i][1][q];
            }
      }
#pragma unroll
      for (int i = 0; i < NC; ++i)
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const int r = g + 8 * (NT == 0 ? e : e >> 1), m = NT == 0 ? t : 8 * i + 2 * t + (e & 1);
          if (r >= nr || m >= M) continue;
          if (direct) {
            s_store<WK, SILU>(a, n0 + row + r, m, acc[0][i][e], acc[WR - 1][i][e]);
          } else {
#pragma unroll
            for (int h = 0; h < WR; ++h) buf[((jj * WR + h) * M + m) * 16 + r] = acc[h][i][e];
          }
        }
    }
    if (direct) continue;
    // the parts (and the cluster's CTAs) of this pass's tiles, in order
    if (a.KS > 1) {
      s_cluster_sync();
    } else {
      __syncthreads();
    }
    const int prows = min(nt * th, rows - t0 * th);
    const int items = prows * M;
    const int ib = rank * items / a.KS, ie = (rank + 1) * items / a.KS;
    for (int it = ib + tid; it < ie; it += NTHR) {
      const int m = it / prows, rr = it - m * prows;  // neighbouring threads: neighbouring outputs
      const int tl = rr / th, r = rr - tl * th;
      const float* p0 = buf + (tl * a.S * WR * M + m) * 16 + r;
      float v = 0.0f, uv = 0.0f;
      for (int q = 0; q < a.KS; ++q) {
#pragma unroll 4
        for (int s = 0; s < a.S; ++s) {
          const float* p = p0 + s * (WR * 16 * M);
          v += a.KS > 1 ? s_ld_rank(p, (uint32_t)q) : *p;
          if constexpr (SILU) uv += a.KS > 1 ? s_ld_rank(p + 16 * M, (uint32_t)q) : p[16 * M];
        }
      }
      s_store<WK, SILU>(a, n0 + t0 * th + rr, m, v, uv);
    }
  }
  __syncthreads();
  if (a.KS > 1) s_cluster_sync();  // no CTA leaves while another reads its partial sums
}

// How many clusters of ks CTAs (one per SM) can run at once: clusters do not
// cross a GPC, so fewer than SMs / ks.
template <int WK, bool SILU, int NT>
cudaError_t s_prepare(int ks, int* n) {
  auto k = stream_linear_kernel<WK, SILU, NT>;
  static std::mutex mu;
  static bool ready[64] = {false};
  static int cache[64][9] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!ready[dev]) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
    ready[dev] = true;
  }
  *n = device_sm_count();
  if (ks == 1) return cudaSuccess;
  if (cache[dev][ks] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ks);
    cfg.blockDim = dim3(32 * s_warps(NT));
    cfg.dynamicSmemBytes = kSmemMax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int c = 0;
    e = cudaOccupancyMaxActiveClusters(&c, k, &cfg);
    if (e != cudaSuccess) return e;
    cache[dev][ks] = c > 0 ? c : 1;
  }
  *n = cache[dev][ks];
  return cudaSuccess;
}

template <int WK, bool SILU, int NT>
cudaError_t s_launch(SArgs a0, cudaStream_t st) {
  constexpr int nw = s_warps(NT);
  a0.U = s_units(WK, a0.K);
  SArgs a = a0;
  int clusters = 0, smem = 0;
  double bt = -1.0;
  for (int ks = 1; ks <= 8; ks *= 2) {
    if (!s_fits(WK, a0.M, a0.K, ks)) continue;
    int n = 0;
    const cudaError_t e = s_prepare<WK, SILU, NT>(ks, &n);
    if (e != cudaSuccess) return e;
    if (n > a0.N) n = (int)a0.N;
    SArgs c = a0;
    c.KS = ks;
    double t = 0.0;
    const int sm = s_split(WK, SILU, nw, n, c, &t);
    if (sm > 0 && (bt < 0.0 || t < bt)) {
      bt = t;
      a = c;
      clusters = n;
      smem = sm;
    }
  }
  if (bt < 0.0) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * a.KS));
  cfg.blockDim = dim3(32 * nw);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (a.KS > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)a.KS;
    at[na].val.clusterDim.y = at[na].val.clusterDim.z = 1;
    ++na;
  }
  const bool legacy = (st == nullptr || st == cudaStreamLegacy || st == cudaStreamPerThread);
  if (!legacy && pdl_enabled()) {
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = at;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, stream_linear_kernel<WK, SILU, NT>, a);
}

template <int WK>
cudaError_t s_launch_wk(const SArgs& a, bool silu, cudaStream_t st) {
  if constexpr (WK == SQ_W_INT4)
    if (a.M == 1) return s_launch<WK, false, 0>(a, st);
  if (a.M <= 8) return silu ? s_launch<WK, true, 1>(a, st) : s_launch<WK, false, 1>(a, st);
  return silu ? s_launch<WK, true, 2>(a, st) : s_launch<WK, false, 2>(a, st);
}

}  // namespace

bool stream_supported(int wkind, int M, int64_t N, int64_t K, int epi) {
  (void)N;
  if (M == 1 && (wkind != SQ_W_INT4 || epi == SQ_EPI_SILU_GATE)) return false;  // not compiled
  for (int ks = 1; ks <= 8; ks *= 2)
    if (s_fits(wkind, M, K, ks)) return true;
  return false;
}

cudaError_t launch_stream(int wkind, const GemvArgs& g, cudaStream_t st) {
  SArgs a = {};
  a.x = g.x;
  a.w = g.w;
  a.scales = g.scales;
  a.bias = g.bias;
  a.residual = g.residual;
  a.y = g.y;
  a.gamma = g.gamma;
  a.eps = g.eps;
  a.M = g.M;
  a.K = (int)g.K;
  a.N = g.N;
  a.row_bytes = g.row_bytes;
  const bool silu = g.epi == SQ_EPI_SILU_GATE;
  switch (wkind) {
    case SQ_W_INT4: return s_launch_wk<SQ_W_INT4>(a, silu, st);
    case SQ_W_FP8: return s_launch_wk<SQ_W_FP8>(a, silu, st);
    default: return s_launch_wk<SQ_W_FP16>(a, silu, st);
  }
}

}  // namespace sq
