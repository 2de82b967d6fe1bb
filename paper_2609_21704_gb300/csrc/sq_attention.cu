// sq_attention.cu -- the decoder around the linear stack: RMSNorm, rotary
// embedding with the KV-cache append, grouped-query decode attention over
// the cache, and the rollback of cache lengths after acceptance.
//
// Sec. III-D.2/3 run the whole model for the draft and verify passes;
// Sec. III-D.4 restarts from the first rejected token, so each model's
// cache keeps only the accepted prefix.  Definitions (no model internals
// are given in the paper; these are the Qwen2.5 decoder's):
//   RMSNorm   y = x / sqrt(mean(x^2) + eps) * gamma       (fp32, fp16 out)
//   RoPE      pairs (d, d + D/2), angle pos * theta^(-2d/D) in 2^-64 turns
//   attention softmax(q . k / sqrt(D)) v over cache positions <= the
//             query's position; query head h reads key/value head
//             h / (Hq / Hkv).
// Layouts: qkv rows [B*T, (Hq + 2 Hkv) D] (q heads, k heads, v heads, the
// fused projection's output); caches [B, Hkv, max_ctx, D] fp16; attention
// output rows [B*T, Hq D].  Token t of sequence b sits at position
// pos0[b] + t.
//
#include <math.h>

#include <mutex>

#include "sq_decoder.h"

namespace sq {

__device__ unsigned int g_attn_status;

constexpr int kHeadDim = 128;
constexpr int kAttnWarps = 4;
constexpr int kAttnThreads = 32 * kAttnWarps;
constexpr int kMaxT = 32;           // new tokens per sequence and call
// Per-query partial record in the workspace: (max, sum, 2 unused, o[D]):
// 132 floats = 528 bytes, so records and their o[] stay 16-byte aligned.
constexpr int kPartStride = kHeadDim + 4;
constexpr int kPartO = 4;

// ---- RMSNorm -----------------------------------------------------------------
__global__ void __launch_bounds__(256) rmsnorm_kernel(const __half* __restrict__ x,
                                                      const __half* __restrict__ gamma, int64_t H,
                                                      float eps, __half* __restrict__ y) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ float red[8];
  const int64_t m = blockIdx.x;
  const __half* xr = x + m * H;
  // sum of squares over 8-value chunks: thread t takes chunks c = t, t + 256,
  // ..., the values of a chunk in order (the order the projections that
  // normalise their own staged rows use, so both give the same bits)
  float ss = 0.0f;
  const int64_t nch = H / 8;
  const bool vec = (reinterpret_cast<uintptr_t>(xr) & 15) == 0;
  for (int64_t c = threadIdx.x; c < nch; c += blockDim.x) {
    if (vec) {
      ss = sumsq8(reinterpret_cast<const uint4*>(xr)[c], ss);
    } else {
      for (int e = 0; e < 8; ++e) {
        const float v = __half2float(xr[8 * c + e]);
        ss = fmaf(v, v, ss);
      }
    }
  }
  if (threadIdx.x == nch % blockDim.x)  // the ragged tail chunk (H % 8 values)
    for (int64_t h = 8 * nch; h < H; ++h) {
      const float v = __half2float(xr[h]);
      ss = fmaf(v, v, ss);
    }
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float t = 0.0f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
  const float r = 1.0f / sqrtf(t / (float)H + eps);
  for (int64_t h = threadIdx.x; h < H; h += blockDim.x)
    y[m * H + h] = __float2half_rn(__half2float(xr[h]) * r * __half2float(gamma[h]));
}

// ---- RoPE --------------------------------------------------------------------
// Inverse frequencies theta^(-2d/D), d < D/2, as turns per position in units
// of 2^-64 of a turn: pos * f modulo 2^64 is the angle modulo 2 pi without
// any fp64 arithmetic (two fp64 operations per clock and SM on this GPU: the
// T positions' table cost 2 us per CTA at T = 28).  f comes from fp64, so
// positions up to 2^17 keep the angle within 1e-10, as an fp64 reduction would.
struct RopeFreq {
  unsigned long long f[kHeadDim / 2];
};

// cos and sin of the angle at `pos`: the turn as a signed fraction a + b of
// 2^64 (24 leading bits, and the rest), times 2 pi in fp32 (head and tail of
// the constant, one rounding of the angle), then fp32 sincosf.
__device__ __forceinline__ float2 rope_cs(int pos, unsigned long long f) {
  const long long turn = (long long)((unsigned long long)(long long)pos * f);
  const float a = __ll2float_rz(turn);
  const float b = __ll2float_rn(turn - __float2ll_rz(a));
  // 2 pi 2^-64 = head + tail
  const float head = 0x1.921fb6p-62f, tail = -0x1.777a5cp-87f;
  const float r = fmaf(a, head, fmaf(a, tail, b * head));
  float s, c;
  sincosf(r, &s, &c);
  return make_float2(c, s);
}

// The rotated pair (x1 c - x2 s, x2 c + x1 s), rounded to fp16 as the cache
// stores it; the products and differences are rounded one by one (no
// contraction), so the separate append and the fused attention write the
// same bits.
__device__ __forceinline__ void rope_rotate_f16(float x1, float x2, float2 cs, __half& y1, __half& y2) {
  y1 = __float2half_rn(__fsub_rn(__fmul_rn(x1, cs.x), __fmul_rn(x2, cs.y)));
  y2 = __float2half_rn(__fadd_rn(__fmul_rn(x2, cs.x), __fmul_rn(x1, cs.y)));
}

// One CTA per (token row, key/value head): rotate the new key, copy the
// value, both into the caches at the token's position.
__global__ void __launch_bounds__(64) kv_append_kernel(const __half* __restrict__ qkv, int T, int Hq,
                                                       int Hkv, const int32_t* __restrict__ pos0,
                                                       const RopeFreq rf, __half* __restrict__ kc,
                                                       __half* __restrict__ vc, int64_t max_ctx) {
  griddep_wait();
  griddep_launch_dependents();
  const int row = blockIdx.x, h = blockIdx.y;
  const int b = row / T, t = row - b * T;
  const int pos = pos0[b] + t;
  if (pos < 0 || (int64_t)pos >= max_ctx) {
    if (threadIdx.x == 0) atomicOr(&g_attn_status, SQ_DEV_BAD_POSITION);
    return;
  }
  const int64_t width = (int64_t)(Hq + 2 * Hkv) * kHeadDim;
  const __half* kr = qkv + row * width + (int64_t)(Hq + h) * kHeadDim;
  const __half* vr = qkv + row * width + (int64_t)(Hq + Hkv + h) * kHeadDim;
  const int64_t dst = (((int64_t)b * Hkv + h) * max_ctx + pos) * kHeadDim;
  const int d = threadIdx.x;  // pair (d, d + D/2)
  const float2 cs = rope_cs(pos, rf.f[d]);
  rope_rotate_f16(__half2float(kr[d]), __half2float(kr[d + kHeadDim / 2]), cs, kc[dst + d],
                  kc[dst + d + kHeadDim / 2]);
  vc[dst + d] = vr[d];
  vc[dst + d + kHeadDim / 2] = vr[d + kHeadDim / 2];
}

// ---- attention ----------------------------------------------------------------
struct AttnArgs {
  const __half* qkv;
  const __half* kc;
  const __half* vc;
  __half* kcw;  // the same caches, written when append != 0
  __half* vcw;
  int append;   // the new tokens' keys/values are appended by the CTAs that hold them
  const int32_t* pos0;
  __half* out;
  float* part;  // [(B*Hkv) * nsplit * Q * kPartStride]: per query (m, l, -, -, o[D]); unused by a cluster
  int B, T, Hq, Hkv, G, Q;
  int64_t max_ctx;
  int nsplit;   // CTAs sharing one (sequence, key/value head, query group)'s keys
  int cluster;  // they form a cluster and merge through distributed shared memory
  float scale;  // 1 / sqrt(D)
  RopeFreq rf;
};

constexpr int kBlockKeys = 64;                         // keys of one pipeline stage
constexpr int kStageHalf = kBlockKeys * kHeadDim * 2;  // bytes of a stage's keys (its values follow)
constexpr float kProbScale = 16384.0f;                 // probabilities enter the product times 2^14

__device__ __forceinline__ void ldsm_x4(uint32_t r[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void attn_mma(float d[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 16-byte asynchronous copy; zeros when !in (src is then not read).
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0)
               : "memory");
}
// Byte offset of 16-byte chunk c of row r in a tile of 256-byte rows: chunks
// are permuted by the row, so the eight rows of a matrix load hit distinct banks.
__device__ __forceinline__ uint32_t tile_off(int r, int c) { return (uint32_t)(r * 256 + ((c ^ (r & 7)) << 4)); }

// (hi, lo): x = hi + lo to 22 bits and more (hi the nearest fp16; a
// non-finite hi carries x alone).
__device__ __forceinline__ void split_f16(float x, __half& hi, __half& lo) {
  hi = __float2half_rn(x);
  const float h = __half2float(hi);
  lo = isfinite(h) ? __float2half_rn(x - h) : __ushort_as_half(0);
}
__device__ __forceinline__ uint32_t pack_h2(__half a, __half b) {
  return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
}

__device__ __forceinline__ uint32_t attn_rank_addr(const float* local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ void attn_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Shapes of the kernel's instances: WM warps along the queries (the other
// kAttnWarps / WM split every block of keys), NT tiles of eight queries a warp.
template <int WM, int NT>
struct AttnCfg {
  static constexpr int kWK = kAttnWarps / WM;          // warps along the keys
  static constexpr int kQT = 8 * WM * NT;              // queries a CTA holds
  static constexpr int kKeysWarp = kBlockKeys / kWK;   // keys of a block a warp takes
  static constexpr int kKeysStep = kKeysWarp < 32 ? kKeysWarp : 32;
  static constexpr int kStages = WM > 1 ? 2 : 3;
  static constexpr int kQBytes = WM * NT * 4096;       // packed query tiles
  static constexpr int kOffFac = kQBytes;              // per query: factor of its scores
  static constexpr int kOffStage = kOffFac + (kQT * 4 + 127) / 128 * 128;
  static constexpr int kOffCs = kOffStage + kStages * 2 * kStageHalf;
};
constexpr int attn_smem(int off_cs, int T) { return off_cs + T * (kHeadDim / 2) * 8; }

// One CTA: kQT queries (q = g * T + t: head kvh * G + g, token t) of one
// (sequence, key/value head) against one contiguous share of its 64-key blocks.
//
// Products on mma.sync (fp16 inputs, fp32 sums; tcgen05 would want 128 query
// rows, these groups have 1 to 200) without giving up fp32 operands: a query
// (rotated in fp32) is split into two fp16 terms after scaling it by a power
// of two (its largest value to [2^10, 2^11)), a probability into two fp16
// terms after scaling by 2^14; keys and values are fp16 already.  An m16 tile
// holds eight queries: rows 0..7 the high terms, rows 8..15 the low terms, so
// both halves of a sum meet in the same lane and small query groups (5 at one
// token of a 40 / 8-head model) waste no second instruction.  Scores, the
// running maximum, probabilities, sums and the weighted values stay fp32
// (online softmax over the blocks).  Keys and values stream through two or
// three stages of 32 KB (cp.async, two CTAs per SM); the number of shares
// depends on the launch (SMs, heads) and their bounds on the device's length,
// so an empty tail of the cache costs nothing.  Bound: cache bytes at one
// token, the doubled products (1021 multiply-adds per clock and SM measured)
// and the exponentials for large query groups.  Measured against the fp32
// CUDA-core kernel over 32-key chunks that this one replaces (append
// included): 4 sequences of 8000 tokens in caches of 16384, 40 / 8 heads, one
// token: 161.7 -> 28.8 us (4.7 TB/s); 28 tokens of 4 sequences behind 2000,
// 28 / 4 heads: 421 -> 65.7 us; error against 64 bits unchanged (2.1e-4, the
// fp16 rounding of the output).
template <int WM, int NT>
__global__ void __launch_bounds__(kAttnThreads, 2) attention_kernel(const AttnArgs a) {
  using C = AttnCfg<WM, NT>;
  constexpr int WK = C::kWK, QT = C::kQT, NJ = C::kKeysStep / 8;
  griddep_wait();
  griddep_launch_dependents();
  extern __shared__ __align__(128) uint8_t asm_[];
  const uint32_t base = smem_u32(asm_);
  float* qfac = reinterpret_cast<float*>(asm_ + C::kOffFac);
  float2* cst = reinterpret_cast<float2*>(asm_ + C::kOffCs);
  const int T = a.T;
  const int bh = (int)(blockIdx.x / (unsigned)a.nsplit), split = (int)(blockIdx.x - (unsigned)bh * a.nsplit);
  const int q0 = blockIdx.y * QT;
  const int b = bh / a.Hkv, kvh = bh - b * a.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p0 = a.pos0[b];
  const int64_t len64 = (int64_t)p0 + T;  // cache entries after the append
  const bool valid = p0 >= 0 && len64 <= a.max_ctx;
  if (a.append && !valid && split == 0 && blockIdx.y == 0 && tid == 0)
    atomicOr(&g_attn_status, SQ_DEV_BAD_POSITION);
  const int len = valid ? (int)len64 : 0;
  const int nblk = (len + kBlockKeys - 1) / kBlockKeys;
  const int blk0 = (int)((int64_t)split * nblk / a.nsplit);
  const int blk1 = (int)((int64_t)(split + 1) * nblk / a.nsplit);
  const int64_t width = (int64_t)(a.Hq + 2 * a.Hkv) * kHeadDim;
  const int64_t cbase = ((int64_t)b * a.Hkv + kvh) * a.max_ctx * kHeadDim;
  const int n_old = a.append ? p0 : len;  // keys read from the caches

  // block -> stage: cached rows by asynchronous copies, rows past the end zero
  auto load_block = [&](int blk, int stage) {
    const uint32_t ks = base + C::kOffStage + stage * 2 * kStageHalf;
#pragma unroll
    for (int i = 0; i < kBlockKeys * 16 / kAttnThreads; ++i) {
      const int idx = tid + i * kAttnThreads;
      const int r = idx >> 4, c = idx & 15;
      const int j = blk * kBlockKeys + r;
      if (j >= n_old && j < len) continue;  // a new key: written by fill_new
      const bool in = j < n_old;
      const int64_t src = cbase + (in ? (int64_t)j * kHeadDim + c * 8 : 0);
      cp16(ks + tile_off(r, c), a.kc + src, in);
      cp16(ks + kStageHalf + tile_off(r, c), a.vc + src, in);
    }
  };
  // append: the new tokens of a block rotated from qkv, used directly and
  // (by the first query group's CTA) written to the caches
  auto fill_new = [&](int blk, int stage) {
    const int j_lo = max(blk * kBlockKeys, n_old), j_hi = min((blk + 1) * kBlockKeys, len);
    uint8_t* ks = asm_ + C::kOffStage + stage * 2 * kStageHalf;
    for (int idx = tid; idx < (j_hi - j_lo) * (kHeadDim / 2); idx += kAttnThreads) {
      const int j = j_lo + idx / (kHeadDim / 2), d = idx % (kHeadDim / 2);
      const int t = j - p0, r = j - blk * kBlockKeys;
      const __half* row = a.qkv + ((int64_t)b * T + t) * width;
      const __half* kr = row + (int64_t)(a.Hq + kvh) * kHeadDim;
      const __half* vr = row + (int64_t)(a.Hq + a.Hkv + kvh) * kHeadDim;
      __half y1, y2;
      rope_rotate_f16(__half2float(kr[d]), __half2float(kr[d + kHeadDim / 2]), cst[t * (kHeadDim / 2) + d], y1, y2);
      const __half v1 = vr[d], v2 = vr[d + kHeadDim / 2];
      const uint32_t o1 = tile_off(r, d >> 3) + (d & 7) * 2;
      const uint32_t o2 = tile_off(r, (d + kHeadDim / 2) >> 3) + (d & 7) * 2;
      *reinterpret_cast<__half*>(ks + o1) = y1;
      *reinterpret_cast<__half*>(ks + o2) = y2;
      *reinterpret_cast<__half*>(ks + kStageHalf + o1) = v1;
      *reinterpret_cast<__half*>(ks + kStageHalf + o2) = v2;
      if (blockIdx.y == 0) {
        const int64_t dst = cbase + (int64_t)j * kHeadDim + d;
        a.kcw[dst] = y1;
        a.kcw[dst + kHeadDim / 2] = y2;
        a.vcw[dst] = v1;
        a.vcw[dst + kHeadDim / 2] = v2;
      }
    }
  };

  // ---- prologue: first blocks requested, then the queries
#pragma unroll
  for (int i = 0; i < C::kStages - 1; ++i) {
    if (blk0 + i < blk1) load_block(blk0 + i, i);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (blk0 < blk1)
    for (int idx = tid; idx < T * (kHeadDim / 2); idx += kAttnThreads)
      cst[idx] = rope_cs(p0 + idx / (kHeadDim / 2), a.rf.f[idx % (kHeadDim / 2)]);
  __syncthreads();
  if (blk0 < blk1) {
    // a warp per query: lane l the pairs (2l, 2l + 64), (2l + 1, 2l + 65)
    const bool qvec = (reinterpret_cast<uintptr_t>(a.qkv) & 3) == 0;
    for (int ql = warp; ql < QT; ql += kAttnWarps) {
      const int q = q0 + ql;
      float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // d = 2l, 2l + 1, 2l + 64, 2l + 65
      if (q < a.Q) {
        const int g = q / T, t = q - g * T;
        const __half* qr = a.qkv + ((int64_t)b * T + t) * width + (int64_t)(kvh * a.G + g) * kHeadDim + 2 * lane;
        float x[4];
        if (qvec) {
          const float2 u1 = __half22float2(*reinterpret_cast<const __half2*>(qr));
          const float2 u2 = __half22float2(*reinterpret_cast<const __half2*>(qr + kHeadDim / 2));
          x[0] = u1.x; x[1] = u1.y; x[2] = u2.x; x[3] = u2.y;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = __half2float(qr[(e & 1) + (e >> 1) * (kHeadDim / 2)]);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float2 cs = cst[t * (kHeadDim / 2) + 2 * lane + e];
          v[e] = x[e] * cs.x - x[e + 2] * cs.y;
          v[e + 2] = x[e + 2] * cs.x + x[e] * cs.y;
        }
      }
      const float am = warp_max(fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3]))));
      int ex = 10;
      if (am > 0.0f && isfinite(am)) ex = max((int)(__float_as_uint(am) >> 23) - 127, -100);
      const float up = __uint_as_float((uint32_t)(127 + 10 - ex) << 23);  // 2^(10 - ex)
      const int tile = ql >> 3, r = ql & 7;
      uint8_t* qt = asm_ + tile * 4096;
      __half hi[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) split_f16(v[e] * up, hi[e], lo[e]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int c = (lane >> 2) + e * 8;
        const uint32_t in = (lane & 3) * 4;
        *reinterpret_cast<uint32_t*>(qt + tile_off(r, c) + in) = pack_h2(hi[2 * e], hi[2 * e + 1]);
        *reinterpret_cast<uint32_t*>(qt + tile_off(r + 8, c) + in) = pack_h2(lo[2 * e], lo[2 * e + 1]);
      }
      if (lane == 0) qfac[ql] = a.scale * __uint_as_float((uint32_t)(127 + ex - 10) << 23);
    }
    if (a.append)
#pragma unroll
      for (int i = 0; i < C::kStages - 1; ++i)
        if (blk0 + i < blk1) fill_new(blk0 + i, i);
  }
  __syncthreads();

  // ---- this warp's share: query tiles wm * NT .. of the CTA, keys
  // [kw * kKeysWarp, + kKeysWarp) of every block
  const int wm = warp % WM, kw = warp / WM;
  const int g = lane >> 2, t4 = lane & 3;
  float o[NT][16][4];
  float mrun[NT], lrun[NT], fac[NT];
  int tpos[NT];  // the query's token
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    mrun[nt] = -INFINITY;
    lrun[nt] = 0.0f;
    const int ql = (wm * NT + nt) * 8 + g;
    fac[nt] = blk0 < blk1 ? qfac[ql] : 0.0f;
    tpos[nt] = (q0 + ql) % T;
#pragma unroll
    for (int i = 0; i < 16; ++i) o[nt][i][0] = o[nt][i][1] = o[nt][i][2] = o[nt][i][3] = 0.0f;
  }
  const uint32_t qbase = base + wm * NT * 4096;
  // matrix-load rows and chunks of this lane: queries (rows 0..15), keys
  // (two eight-key tiles), values (transposed)
  const int qrow = (lane & 7) + ((lane >> 3) & 1) * 8, qch = lane >> 4;
  const int krow = (lane & 7) + (lane >> 4) * 8, kch = (lane >> 3) & 1;
  const int vrow = (lane & 7) + ((lane >> 3) & 1) * 8, vch = lane >> 4;
  uint32_t qreg[NT == 1 ? 8 : 1][4];
  if constexpr (NT == 1) {
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) ldsm_x4(qreg[kk], qbase + tile_off(qrow, 2 * kk + qch));
  }

  for (int blk = blk0; blk < blk1; ++blk) {
    const int it = blk - blk0;
    asm volatile("cp.async.wait_group %0;" ::"n"(C::kStages - 2) : "memory");
    __syncthreads();
    {
      const int nx = blk + C::kStages - 1;
      if (nx < blk1) {
        load_block(nx, (it + C::kStages - 1) % C::kStages);
        if (a.append && (nx + 1) * kBlockKeys > n_old) fill_new(nx, (it + C::kStages - 1) % C::kStages);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const uint32_t ks = base + C::kOffStage + (it % C::kStages) * 2 * kStageHalf;
    const uint32_t vs = ks + kStageHalf;
    const bool edge = (blk + 1) * kBlockKeys > p0;  // some key may lie past a query
#pragma unroll 1
    for (int sub = 0; sub < C::kKeysWarp / C::kKeysStep; ++sub) {
      const int kb = kw * C::kKeysWarp + sub * C::kKeysStep;
      float s[NT][NJ][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int j = 0; j < NJ; ++j) s[nt][j][0] = s[nt][j][1] = s[nt][j][2] = s[nt][j][3] = 0.0f;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        uint32_t qa[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          if constexpr (NT == 1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) qa[0][e] = qreg[kk][e];
          } else {
            ldsm_x4(qa[nt], qbase + nt * 4096 + tile_off(qrow, 2 * kk + qch));
          }
        }
#pragma unroll
        for (int jp = 0; jp < NJ / 2; ++jp) {
          uint32_t kf[4];
          ldsm_x4(kf, ks + tile_off(kb + jp * 16 + krow, 2 * kk + kch));
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            attn_mma(s[nt][2 * jp], qa[nt], kf[0], kf[1]);
            attn_mma(s[nt][2 * jp + 1], qa[nt], kf[2], kf[3]);
          }
        }
      }
      // scores (high + low terms), mask, running maximum, probabilities
      uint32_t pa[NT][NJ / 2][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            // (an infinite key: the high term alone has the sign)
            const float sl = s[nt][j][e + 2];
            float v = (s[nt][j][e] + (fabsf(sl) < INFINITY ? sl : 0.0f)) * fac[nt];
            if (edge && blk * kBlockKeys + kb + 8 * j + 2 * t4 + e > p0 + tpos[nt]) v = -INFINITY;
            s[nt][j][e] = v;
            mx = fmaxf(mx, v);
          }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float mnew = fmaxf(mrun[nt], mx);
        if (__any_sync(0xffffffffu, mnew > mrun[nt])) {
          const float corr = mrun[nt] == -INFINITY ? 0.0f : expf(mrun[nt] - mnew);
          lrun[nt] *= corr;
#pragma unroll
          for (int i = 0; i < 16; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[nt][i][e] *= corr;
          mrun[nt] = mnew;
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          __half hi[2], lo[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float p = mrun[nt] == -INFINITY ? 0.0f : expf(s[nt][j][e] - mrun[nt]);
            lrun[nt] += p;
            split_f16(p * kProbScale, hi[e], lo[e]);
          }
          pa[nt][j >> 1][(j & 1) * 2] = pack_h2(hi[0], hi[1]);
          pa[nt][j >> 1][(j & 1) * 2 + 1] = pack_h2(lo[0], lo[1]);
        }
      }
#pragma unroll
      for (int jj = 0; jj < NJ / 2; ++jj)
#pragma unroll
        for (int dp = 0; dp < 8; ++dp) {
          uint32_t vf[4];
          ldsm_x4_t(vf, vs + tile_off(kb + jj * 16 + vrow, 2 * dp + vch));
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            attn_mma(o[nt][2 * dp], pa[nt][jj], vf[0], vf[1]);
            attn_mma(o[nt][2 * dp + 1], pa[nt][jj], vf[2], vf[3]);
          }
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  // ---- this CTA's partial records (m, l, -, -, o[D]) in shared memory, over
  // the stages: one per warp first, then the warps along the keys in order
  float* rec = reinterpret_cast<float*>(asm_ + C::kOffStage);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    float l = lrun[nt];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    float* r = rec + ((kw * WM + wm) * NT * 8 + nt * 8 + g) * kPartStride;
    if (t4 == 0) {
      r[0] = mrun[nt];
      r[1] = l;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      // (an infinite value: the high term alone has the sign)
      const float l0 = fabsf(o[nt][i][2]) < INFINITY ? o[nt][i][2] : 0.0f;
      const float l1 = fabsf(o[nt][i][3]) < INFINITY ? o[nt][i][3] : 0.0f;
      const float2 v = make_float2((o[nt][i][0] + l0) * (1.0f / kProbScale), (o[nt][i][1] + l1) * (1.0f / kProbScale));
      *reinterpret_cast<float2*>(r + kPartO + 8 * i + 2 * t4) = v;
    }
  }
  __syncthreads();
  const int nq = min(QT, a.Q - q0);
  float* mine = WK > 1 ? rec + WK * QT * kPartStride : rec;
  if constexpr (WK > 1) {
    for (int idx = tid; idx < nq * (kHeadDim / 4); idx += kAttnThreads) {
      const int q = idx / (kHeadDim / 4), d4 = idx % (kHeadDim / 4);
      float M = -INFINITY;
#pragma unroll
      for (int w = 0; w < WK; ++w) M = fmaxf(M, rec[(w * QT + q) * kPartStride]);
      float L = 0.0f;
      float4 O = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (M != -INFINITY)
#pragma unroll
        for (int w = 0; w < WK; ++w) {
          const float* r = rec + (w * QT + q) * kPartStride;
          if (r[0] == -INFINITY) continue;
          const float f = expf(r[0] - M);
          const float4 v = *reinterpret_cast<const float4*>(r + kPartO + 4 * d4);
          L = fmaf(f, r[1], L);
          O.x = fmaf(f, v.x, O.x);
          O.y = fmaf(f, v.y, O.y);
          O.z = fmaf(f, v.z, O.z);
          O.w = fmaf(f, v.w, O.w);
        }
      float* r = mine + q * kPartStride;
      if (d4 == 0) {
        r[0] = M;
        r[1] = L;
      }
      *reinterpret_cast<float4*>(r + kPartO + 4 * d4) = O;
    }
    __syncthreads();
  }

  if (!a.cluster && a.nsplit > 1) {  // records to the workspace, merged by attention_combine_kernel
    float* part = a.part + (((int64_t)bh * a.nsplit + split) * a.Q + q0) * kPartStride;
    for (int idx = tid; idx < nq * (kPartStride / 4); idx += kAttnThreads)
      reinterpret_cast<float4*>(part)[idx] = reinterpret_cast<const float4*>(mine)[idx];
    return;
  }
  // ---- the cluster's records merged in rank order; rank r writes its share
  const int S = a.nsplit;
  if (S > 1) attn_cluster_sync();
  const int items = nq * (kHeadDim / 4);
  const int i0 = (int)((int64_t)split * items / S), i1 = (int)((int64_t)(split + 1) * items / S);
  const bool ovec = (reinterpret_cast<uintptr_t>(a.out) & 7) == 0;
  for (int idx = i0 + tid; idx < i1; idx += kAttnThreads) {
    const int q = idx / (kHeadDim / 4), d4 = idx % (kHeadDim / 4);
    float M = -INFINITY, L = 0.0f;
    float4 O = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int s0 = 0; s0 < S; s0 += 8) {
      // eight ranks' records in flight, then added in rank order
      float4 ml[8], ov[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (s0 + u < S) {
          const uint32_t r = S > 1 ? attn_rank_addr(mine + q * kPartStride, (uint32_t)(s0 + u))
                                   : smem_u32(mine + q * kPartStride);
          ml[u] = ld_cluster_f4(r);
          ov[u] = ld_cluster_f4(r + (kPartO + 4 * d4) * 4);
        }
      float Mn = M;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (s0 + u < S) Mn = fmaxf(Mn, ml[u].x);
      if (Mn == -INFINITY) continue;
      const float c = M == -INFINITY ? 0.0f : expf(M - Mn);
      L *= c;
      O.x *= c; O.y *= c; O.z *= c; O.w *= c;
      M = Mn;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (s0 + u < S && ml[u].x != -INFINITY) {
          const float f = expf(ml[u].x - M);
          L = fmaf(f, ml[u].y, L);
          O.x = fmaf(f, ov[u].x, O.x);
          O.y = fmaf(f, ov[u].y, O.y);
          O.z = fmaf(f, ov[u].z, O.z);
          O.w = fmaf(f, ov[u].w, O.w);
        }
    }
    const int qq = q0 + q, hg = qq / T, t = qq - hg * T;
    __half* dst = a.out + (((int64_t)b * T + t) * a.Hq + kvh * a.G + hg) * kHeadDim + 4 * d4;
    const __half h0 = __float2half_rn(L > 0.0f ? O.x / L : 0.0f), h1 = __float2half_rn(L > 0.0f ? O.y / L : 0.0f);
    const __half h2 = __float2half_rn(L > 0.0f ? O.z / L : 0.0f), h3 = __float2half_rn(L > 0.0f ? O.w / L : 0.0f);
    if (ovec) {
      *reinterpret_cast<uint2*>(dst) = make_uint2(pack_h2(h0, h1), pack_h2(h2, h3));
    } else {
      dst[0] = h0; dst[1] = h1; dst[2] = h2; dst[3] = h3;
    }
  }
  __syncthreads();
  if (S > 1) attn_cluster_sync();  // no CTA leaves while another reads its records
}

// One CTA per (sequence and key/value head, query): the chunk maxima and
// sums are read in parallel into shared memory, then each thread (one per
// head dimension) merges the chunks' weighted values.
__global__ void __launch_bounds__(kHeadDim) attention_combine_kernel(const AttnArgs a) {
  griddep_wait();
  griddep_launch_dependents();
  extern __shared__ float cm[];  // [2 * nsplit]: chunk max, chunk sum
  __shared__ float red[kHeadDim / 32];
  const int bh = blockIdx.x, q = blockIdx.y, d = threadIdx.x;
  const int b = bh / a.Hkv, kvh = bh - b * a.Hkv;
  const float* base = a.part + (int64_t)bh * a.nsplit * a.Q * kPartStride;
  float M = -INFINITY;
  for (int s = d; s < a.nsplit; s += kHeadDim) {
    const float* ps = base + ((int64_t)s * a.Q + q) * kPartStride;
    cm[s] = ps[0];
    cm[a.nsplit + s] = ps[1];
    M = fmaxf(M, ps[0]);
  }
  M = warp_max(M);
  if ((d & 31) == 0) red[d >> 5] = M;
  __syncthreads();
  M = -INFINITY;
#pragma unroll
  for (int w = 0; w < kHeadDim / 32; ++w) M = fmaxf(M, red[w]);
  float L = 0.0f, O = 0.0f;
  if (M != -INFINITY)
    for (int s0 = 0; s0 < a.nsplit; s0 += 8) {
      // the chunks' weighted values, eight loads in flight; then the same
      // sums, chunk by chunk in order
      float ov[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int s = s0 + u;
        ov[u] = (s < a.nsplit && cm[s] != -INFINITY) ? base[((int64_t)s * a.Q + q) * kPartStride + kPartO + d]
                                                      : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int s = s0 + u;
        if (s >= a.nsplit) break;
        const float ms = cm[s];
        if (ms == -INFINITY) continue;
        const float w = expf(ms - M);
        L = fmaf(w, cm[a.nsplit + s], L);
        O = fmaf(w, ov[u], O);
      }
    }
  const int g = q / a.T, t = q - g * a.T;
  const int64_t row = (int64_t)b * a.T + t;
  a.out[row * (int64_t)a.Hq * kHeadDim + (int64_t)(kvh * a.G + g) * kHeadDim + d] =
      __float2half_rn(L > 0.0f ? O / L : 0.0f);
}

// ---- embedding ---------------------------------------------------------------------
// out[m, :] = table[ids[m], :] (fp16 copy, 16-byte pieces when aligned); an id
// outside [0, V) gives a zero row and sets SQ_DEV_BAD_TOKEN_ID.
__global__ void __launch_bounds__(256) embed_kernel(const int32_t* __restrict__ ids, int64_t ids_stride,
                                                    const __half* __restrict__ table, int64_t V,
                                                    int64_t H, __half* __restrict__ out) {
  griddep_wait();
  griddep_launch_dependents();
  const int64_t m = blockIdx.x;
  const int32_t id = ids[m * ids_stride];
  const bool ok = id >= 0 && (int64_t)id < V;
  if (!ok && threadIdx.x == 0) atomicOr(&g_attn_status, SQ_DEV_BAD_TOKEN_ID);
  const __half* src = table + (ok ? (int64_t)id : 0) * H;
  __half* dst = out + m * H;
  if ((H & 7) == 0 && ((reinterpret_cast<uintptr_t>(table) | reinterpret_cast<uintptr_t>(out)) & 15) == 0) {
    for (int64_t i = threadIdx.x; i < H / 8; i += blockDim.x)
      reinterpret_cast<uint4*>(dst)[i] = ok ? reinterpret_cast<const uint4*>(src)[i] : make_uint4(0, 0, 0, 0);
  } else {
    for (int64_t i = threadIdx.x; i < H; i += blockDim.x) dst[i] = ok ? src[i] : __ushort_as_half(0);
  }
}

cudaError_t launch_embed(const int32_t* ids, int M, int64_t ids_stride, const __half* table, int64_t V,
                         int64_t H, __half* out, cudaStream_t st) {
  if (M == 0) return cudaSuccess;
  return launch_pdl(embed_kernel, dim3((unsigned)M), dim3(256), 0, st, ids, ids_stride, table, V, H, out);
}

// ---- speculative bookkeeping (Sec. III-D.4: the accepted prefix plus the
// correction becomes the context of the next cycle) ----------------------------------
// One thread per sequence.  Appends the n + 1 committed tokens to the history
// and derives the next cycle's inputs: the positions of the K draft steps and
// of the verify pass, and the last two committed tokens (the draft's first
// step re-reads the second-last one, whose key/value the draft may not have
// computed when every draft was accepted).
__global__ void spec_commit_kernel(const int32_t* __restrict__ n_acc, const int32_t* __restrict__ tokens,
                                   int ldt, int B, int K, int32_t* __restrict__ hist, int cap,
                                   int32_t* __restrict__ len, int32_t* __restrict__ pos,
                                   int32_t* __restrict__ last2) {
  griddep_wait();
  griddep_launch_dependents();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  int L = len[b];
  int32_t* h = hist + (int64_t)b * cap;
  bool bad = L < 0 || L > cap;
  if (!bad) {
    const int na = n_acc ? n_acc[b] : 0;
    if (na >= ldt) {
      bad = true;
    } else if (na >= 0) {
      const int cnt = na + 1 < cap - L ? na + 1 : cap - L;
      for (int i = 0; i < cnt; ++i) h[L + i] = tokens[(int64_t)b * ldt + i];
      if (cnt < na + 1) bad = true;
      L += cnt;
    }
  }
  if (bad || L < 2) {
    atomicOr(&g_attn_status, SQ_DEV_BAD_POSITION);
    if (L < 0 || L > cap) L = 0;
  }
  len[b] = L;
  last2[2 * b] = L >= 2 ? h[L - 2] : -1;
  last2[2 * b + 1] = L >= 1 ? h[L - 1] : -1;
  if (K >= 1) pos[b] = L - 2;
  for (int k = 1; k < K; ++k) pos[(int64_t)k * B + b] = L - 1 + k;
  pos[(int64_t)K * B + b] = L - 1;
}

// verify_tokens[b, :] = (last committed token, draft 1 .. K); draft[b, k] =
// samples[k, b] (the draft steps write one token per sequence).
__global__ void spec_drafts_kernel(const int32_t* __restrict__ samples, const int32_t* __restrict__ last2,
                                   int B, int K, int32_t* __restrict__ verify, int32_t* __restrict__ draft) {
  griddep_wait();
  griddep_launch_dependents();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  verify[(int64_t)b * (K + 1)] = last2[2 * b + 1];
  for (int k = 0; k < K; ++k) {
    const int32_t t = samples[(int64_t)k * B + b];
    verify[(int64_t)b * (K + 1) + 1 + k] = t;
    draft[(int64_t)b * K + k] = t;
  }
}

cudaError_t launch_spec_commit(const int32_t* n, const int32_t* tokens, int ldt, int B, int K, int32_t* hist,
                               int cap, int32_t* len, int32_t* pos, int32_t* last2, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  return launch_pdl(spec_commit_kernel, dim3((unsigned)((B + 127) / 128)), dim3(128), 0, st, n, tokens, ldt,
                    B, K, hist, cap, len, pos, last2);
}

cudaError_t launch_spec_drafts(const int32_t* samples, const int32_t* last2, int B, int K, int32_t* verify,
                               int32_t* draft, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  return launch_pdl(spec_drafts_kernel, dim3((unsigned)((B + 127) / 128)), dim3(128), 0, st, samples, last2,
                    B, K, verify, draft);
}

// ---- rollback -------------------------------------------------------------------
__global__ void kv_rollback_kernel(const int32_t* __restrict__ base, const int32_t* __restrict__ n,
                                   int B, int limit, int32_t* __restrict__ len) {
  griddep_wait();
  griddep_launch_dependents();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int na = n[b];
  len[b] = na < 0 ? base[b] : base[b] + (na + 1 < limit ? na + 1 : limit);
}

// ---- host side -------------------------------------------------------------------
cudaError_t launch_rmsnorm(const __half* x, const __half* gamma, int M, int64_t H, float eps, __half* y,
                           cudaStream_t st) {
  if (M == 0) return cudaSuccess;
  return launch_pdl(rmsnorm_kernel, dim3((unsigned)M), dim3(256), 0, st, x, gamma, H, eps, y);
}

static RopeFreq rope_freq(double theta) {
  // the last theta's table per host thread (64 pow calls take longer than a launch)
  static thread_local double last = 0.0;
  static thread_local RopeFreq rf;
  if (theta != last) {
    for (int d = 0; d < kHeadDim / 2; ++d) {
      const double turns = pow(theta, -2.0 * d / (double)kHeadDim) / 6.283185307179586;
      rf.f[d] = (unsigned long long)(turns * 18446744073709551616.0);
    }
    last = theta;
  }
  return rf;
}

cudaError_t launch_kv_append(const __half* qkv, int B, int T, int Hq, int Hkv, const int32_t* pos0,
                             double theta, __half* kc, __half* vc, int64_t max_ctx, cudaStream_t st) {
  if (B == 0 || T == 0) return cudaSuccess;
  return launch_pdl(kv_append_kernel, dim3((unsigned)(B * T), (unsigned)Hkv), dim3(kHeadDim / 2), 0, st,
                    qkv, T, Hq, Hkv, pos0, rope_freq(theta), kc, vc, max_ctx);
}

// Room for one record per query and 32 cache positions (more than the shares
// of 64-key blocks ever need).
size_t attention_workspace_bytes(int B, int T, int Hq, int Hkv, int64_t max_ctx) {
  if (B < 0 || T < 0 || Hkv <= 0 || max_ctx <= 0) return 0;
  const int64_t nsplit = (max_ctx + 31) / 32;
  const int64_t Q = (int64_t)(Hq / Hkv) * T;
  return (size_t)B * Hkv * nsplit * Q * kPartStride * sizeof(float);
}

int attention_max_tokens() { return kMaxT; }

constexpr int kAttnMaxCluster = 16;
constexpr int kTwoPerSmTokens = 24;  // new tokens up to which two CTAs of every instance share an SM
constexpr int kShortBlocks = 8;

// Prepares an instance and returns how many clusters of S of its CTAs can be
// resident (cached per device, S and shared memory of up to kTwoPerSmTokens or
// kMaxT new tokens; S = 0: only prepares).
template <int WM, int NT>
static cudaError_t attn_resident(int S, int T, int* n) {
  auto k = attention_kernel<WM, NT>;
  constexpr int kSmem[2] = {attn_smem(AttnCfg<WM, NT>::kOffCs, kTwoPerSmTokens),
                            attn_smem(AttnCfg<WM, NT>::kOffCs, kMaxT)};
  static std::mutex mu;
  static bool ready[64] = {false};
  static int cache[64][2][kAttnMaxCluster + 1] = {};
  const int wide = T > kTwoPerSmTokens;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!ready[dev]) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem[1]);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    ready[dev] = true;
  }
  if (S == 0) return cudaSuccess;
  if (cache[dev][wide][S] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)S);
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = (size_t)kSmem[wide];
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)S;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int c = 0;
    if (cudaOccupancyMaxActiveClusters(&c, k, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      c = 0;
    }
    cache[dev][wide][S] = c + 1;
  }
  *n = cache[dev][wide][S] - 1;
  return cudaSuccess;
}

// How many CTAs share the keys of one (sequence, key/value head, query
// group), and how they meet.  As many as fill the two CTAs per SM, at most
// one per 64-key block of the cache; up to 16 meet in a cluster (one launch,
// the records never leave the chip), as long as all clusters are resident at
// once.  A long cache under few heads wants more shares than that: from 16
// blocks a CTA on, the records go through the workspace and a second launch
// merges them.
template <int WM, int NT>
static cudaError_t launch_attn_inst(AttnArgs a, cudaStream_t st) {
  using C = AttnCfg<WM, NT>;
  const int smem = attn_smem(C::kOffCs, a.T);
  const int Z = (a.Q + C::kQT - 1) / C::kQT;
  const int64_t base = (int64_t)a.B * a.Hkv * Z;
  const int64_t blocks = (a.max_ctx + kBlockKeys - 1) / kBlockKeys;
  int64_t S = 2 * (int64_t)device_sm_count() / base;
  if (S > blocks) S = blocks;
  if (S < 1) S = 1;
  a.cluster = S > 1 && (S <= kAttnMaxCluster || blocks <= kAttnMaxCluster * 16);
  int n = 0;
  cudaError_t e = attn_resident<WM, NT>(0, a.T, &n);
  if (e != cudaSuccess) return e;
  if (a.cluster) {
    if (S > kAttnMaxCluster) S = kAttnMaxCluster;
    for (; S > 1; --S) {
      e = attn_resident<WM, NT>((int)S, a.T, &n);
      if (e != cudaSuccess) return e;
      if (n >= base) break;
    }
    a.cluster = S > 1;
  }
  a.nsplit = (int)S;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(S * a.B * a.Hkv), (unsigned)Z);
  cfg.blockDim = dim3(kAttnThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (a.cluster) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)S;
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
  e = cudaLaunchKernelEx(&cfg, attention_kernel<WM, NT>, a);
  if (e != cudaSuccess || a.cluster || S == 1) return e;
  return launch_pdl(attention_combine_kernel, dim3((unsigned)(a.B * a.Hkv), (unsigned)a.Q), dim3(kHeadDim),
                    (size_t)2 * a.nsplit * sizeof(float), st, a);
}

cudaError_t launch_attention(const __half* qkv, int B, int T, int Hq, int Hkv, const int32_t* pos0,
                             double theta, const __half* kc, const __half* vc, int64_t max_ctx,
                             __half* out, void* ws, cudaStream_t st, __half* kc_append,
                             __half* vc_append) {
  if (B == 0 || T == 0) return cudaSuccess;
  AttnArgs a = {};
  a.qkv = qkv;
  a.kc = kc;
  a.vc = vc;
  a.kcw = kc_append;
  a.vcw = vc_append;
  a.append = kc_append != nullptr && vc_append != nullptr;
  a.pos0 = pos0;
  a.out = out;
  a.part = reinterpret_cast<float*>(ws);
  a.B = B;
  a.T = T;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.G = Hq / Hkv;
  a.Q = a.G * T;
  a.max_ctx = max_ctx;
  a.rf = rope_freq(theta);
  a.scale = 1.0f / sqrtf((float)kHeadDim);
  // Instances by the group's queries, so that the keys are read once a group.
  // A cache of at most kShortBlocks blocks has no keys to share out, and a CTA's
  // time is its chain of queries: there eight queries a CTA while those CTAs are
  // resident at once (one block, above 32 queries: two rounds of them still are
  // faster; above kTwoPerSmTokens one such CTA fills an SM).  Cache of 64, 28 / 4
  // heads, 7 tokens: 1 sequence 21.5 -> 7.2 us, 16 sequences 21.8 -> 14.4; cache
  // of 512, 40 / 8 heads, 4 tokens: 10.8 -> 7.8.  20 tokens of 16 sequences, 8 / 8
  // heads (384 CTAs of 32 queries at most): 13.9, with eight 16.0.
  const int64_t blocks = (max_ctx + kBlockKeys - 1) / kBlockKeys;
  const int64_t sms = device_sm_count(), groups = (int64_t)B * Hkv * ((a.Q + 7) / 8);
  const bool few = blocks <= kShortBlocks && (T <= kTwoPerSmTokens ? groups <= (blocks == 1 && a.Q > 32 ? 4 : 2) * sms
                                                                   : groups * blocks <= sms);
  if (a.Q <= 8 || few) return launch_attn_inst<1, 1>(a, st);
  if (a.Q <= 16) return launch_attn_inst<1, 2>(a, st);
  if (a.Q <= 32) return launch_attn_inst<2, 2>(a, st);
  return launch_attn_inst<4, 2>(a, st);
}

cudaError_t launch_kv_rollback(const int32_t* base, const int32_t* n, int B, int limit, int32_t* len,
                               cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  return launch_pdl(kv_rollback_kernel, dim3((unsigned)((B + 127) / 128)), dim3(128), 0, st, base, n, B,
                    limit, len);
}

cudaError_t take_attn_status(uint32_t* bits) {
  uint32_t v = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_attn_status, sizeof(v));
  if (e != cudaSuccess) return e;
  if (v) e = cudaMemcpyToSymbol(g_attn_status, &zero, sizeof(zero));
  *bits |= v;
  return e;
}

}  // namespace sq
