// sq_quantize.cu -- derive the draft variants from the FP16 parent.
//
// Sec. III-A.1: Q4 = f(W16, 4).  Sec. III-A.2: Q8 = f(W16, 8).  The paper
// names no scheme; the one implemented (and documented in specquant.h):
//   INT4: per 128-wide group along K, s = fp16(fp32(amax / 7)) (2^-24 if
//         that rounds to zero for amax > 0), c = clamp(rint(w / s), -8, 7).
//   FP8:  per output row, s = fp32(amax / 448), code = E4M3_satfinite(w / s).
// Every division is the IEEE fp32 divide (__fdiv_rn) and every rounding is
// to nearest even, so codes and scales are bit-identical to the definition.
// These kernels never let the next kernel start early: linear kernels read
// their weights before waiting on the previous kernel, and the weights may
// be what this kernel writes.
//
// The quotients: the IEEE divide costs a dozen instructions, so w / s is
// bracketed instead.  With r = fp32(1 / s), w r (1 -+ 2^-21) lie on either
// side of fp32(w / s) (r and each product are within 2^-24 of exact); where
// both round to the same code, that is the code.  Where they do not (exact
// ties of INT4 codes, about 3 in 10^4 Gaussian weights; next to none of FP8),
// the thread divides.
//
// Bound: HBM, 2 B read per weight, 0.516 B (INT4) or 1 B (FP8) written.
#include "sq_internal.h"

namespace sq {

__device__ unsigned int g_quant_status;

constexpr int kQuantThreads = 256;

__device__ __forceinline__ void halves8(const uint4 v, float out[8]) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&u[i]));
    out[2 * i] = f.x;
    out[2 * i + 1] = f.y;
  }
}

// Largest magnitude of eight fp16 values as fp16 bits (which order like
// integers; 0x7c00 and up: an infinity or NaN among them).
__device__ __forceinline__ uint32_t absmax8(const uint4 v, uint32_t m) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t a = u[i] & 0x7fff7fffu;
    m = __vmaxu2(m, a);  // per half
  }
  return m;
}

// The definition's INT4 code (plus 8) by division.
__device__ __forceinline__ uint32_t int4_code(float w, float s) {
  if (s == 0.0f) return 8u;
  return (uint32_t)((int)fminf(fmaxf(rintf(__fdiv_rn(w, s)), -8.0f), 7.0f) + 8);
}

// A warp takes 1024 consecutive weights (PER = 4), eight groups, as four coalesced
// 16-byte loads a lane (lane l holds chunk 32 i + l: sixteen lanes a group and
// load).  The maxima of a lane's four groups are reduced together, packed in
// pairs; lane j mod 4 then divides for group j only, so a group's two divides
// cost a quarter of a lane's issue slots.  The 14B fused gate/up (27648 x
// 5120) takes 73 us, 4.9 TB/s of the measured 6.8; one lane per four weights
// with a divide per weight took 214.  Bound: about half issue slots (7 a
// weight), half memory.
// PER = 1: 256 weights a warp, for matrices that leave SMs without one otherwise
// (100 x 1024: 2.9 us with four, 2.1 with one).
template <int PER>
__global__ void __launch_bounds__(kQuantThreads) quant_int4_kernel(const __half* __restrict__ w, int64_t N,
                                                                   int64_t K, uint8_t* __restrict__ codes,
                                                                   __half* __restrict__ scales) {
  griddep_wait();  // no early trigger: a linear call may read these outputs at once
  const int lane = threadIdx.x & 31;
  const int64_t total = N * (K / 8);  // chunks; a row is whole groups of 16, so groups are contiguous
  const int64_t step = (int64_t)gridDim.x * (kQuantThreads / 32) * 32 * PER;
  const int64_t wid = (int64_t)blockIdx.x * (kQuantThreads / 32) + (threadIdx.x >> 5);
  for (int64_t c0 = wid * 32 * PER; c0 < total; c0 += step) {
    uint4 v[PER];
    uint32_t m[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int64_t c = c0 + 32 * i + lane;  // the lanes of a group are in or out together
      v[i] = c < total ? ld_stream16(w + 8 * c) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      m[i] = absmax8(v[i], 0u);
      m[i] = max(m[i] & 0xffffu, m[i] >> 16);
    }
    // this lane's group: load lane mod PER, half-warp lane >> 4
    uint32_t mine;
    if constexpr (PER == 4) {
      uint32_t pk[2] = {m[0] | (m[1] << 16), m[2] | (m[3] << 16)};
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        pk[0] = __vmaxu2(pk[0], __shfl_xor_sync(0xffffffffu, pk[0], o));
        pk[1] = __vmaxu2(pk[1], __shfl_xor_sync(0xffffffffu, pk[1], o));
      }
      mine = ((lane & 2 ? pk[1] : pk[0]) >> (16 * (lane & 1))) & 0xffffu;
    } else {
      mine = m[0];
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) mine = max(mine, __shfl_xor_sync(0xffffffffu, mine, o));
    }
    const bool bad = mine >= 0x7c00u;
    float amax = __half2float(__ushort_as_half((uint16_t)mine));
    if (__any_sync(0xffffffffu, bad)) {
      // the largest magnitude that is not NaN, as fmaxf takes it
      float keep = amax;
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        float f[8], a = 0.0f;
        halves8(v[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) a = fmaxf(a, fabsf(f[e]));
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
        if (lane % PER == i) keep = a;
      }
      amax = keep;
      if (bad && (lane & 15) < PER) atomicOr(&g_quant_status, SQ_DEV_NONFINITE_WEIGHT);
    }
    __half sh = __float2half_rn(__fdiv_rn(amax, 7.0f));
    if (amax > 0.0f && __half_as_ushort(sh) == 0) sh = __ushort_as_half(1);
    const float s = __half2float(sh);
    // -1: the codes by division (below the normal scales a code can pass 7)
    const float r = bad || s < 0x1p-14f ? -1.0f : __fdiv_rn(1.0f, s);
    if ((lane & 15) < PER) {
      const int64_t g = (c0 >> 4) + 2 * (lane % PER) + (lane >> 4);
      if (g < (total >> 4)) scales[g] = sh;
    }
    // codes by bracketing: fma(w, r, magic) rounds the quotient into the low
    // bits of the sum, the integer sums of those bits (shifted) place the nibbles
    const float magic = 12582912.0f + 8.0f;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int src = (lane & 16) | i;
      const float gs = __shfl_sync(0xffffffffu, s, src), gr = __shfl_sync(0xffffffffu, r, src);
      const float rlo = gr * (1.0f - 0x1p-21f), rhi = gr * (1.0f + 0x1p-21f);
      float f[8];
      halves8(v[i], f);
      uint32_t acc = 0, diff = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t lo = __float_as_uint(fmaf(f[e], rlo, magic)), hi = __float_as_uint(fmaf(f[e], rhi, magic));
        diff |= lo ^ hi;
        acc += lo << (4 * e);
      }
      uint32_t word = acc - 0x4b400000u * 0x11111111u;  // the exponent bits of the eight sums
      if (diff != 0 || gr < 0.0f) {
        word = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) word |= int4_code(f[e], gs) << (4 * e);
      }
      const int64_t c = c0 + 32 * i + lane;
      if (c < total) reinterpret_cast<uint32_t*>(codes)[c] = word;
    }
  }
}

// Codes of eight weights of an FP8 row.
__device__ __forceinline__ uint2 fp8_codes8(const uint4 v, float s, float rlo, float rhi) {
  float f[8];
  halves8(v, f);
  uint32_t lo[2] = {0u, 0u}, hi[2] = {0u, 0u};
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    lo[e >> 2] |= (uint32_t)f32x2_to_e4m3x2(f[e] * rlo, f[e + 1] * rlo) << (8 * (e & 3));
    hi[e >> 2] |= (uint32_t)f32x2_to_e4m3x2(f[e] * rhi, f[e + 1] * rhi) << (8 * (e & 3));
  }
  // (a row without a scale: every code is +0, also that of a NaN, whose bounds agree)
  if (((lo[0] ^ hi[0]) | (lo[1] ^ hi[1])) != 0u || s == 0.0f) {
    lo[0] = lo[1] = 0u;
    if (s != 0.0f)
#pragma unroll
      for (int e = 0; e < 8; e += 2)
        lo[e >> 2] |= (uint32_t)f32x2_to_e4m3x2(__fdiv_rn(f[e], s), __fdiv_rn(f[e + 1], s)) << (8 * (e & 3));
  }
  return make_uint2(lo[0], lo[1]);
}

// A group of TPR threads per row: its first kFp8Keep chunks of eight weights
// per thread stay in registers between the maximum and the codes, longer rows
// read the rest again.
constexpr int kFp8Keep = 8;
template <int TPR>
__global__ void __launch_bounds__(kQuantThreads) quant_fp8_kernel(const __half* __restrict__ w, int64_t N,
                                                                  int64_t K, uint8_t* __restrict__ codes,
                                                                  float* __restrict__ scales) {
  griddep_wait();  // no early trigger: a linear call may read these outputs at once
  constexpr int RPC = kQuantThreads / TPR;  // rows a CTA holds at once
  __shared__ uint32_t red[2][kQuantThreads / 32];
  __shared__ float redf[2][kQuantThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rt = threadIdx.x % TPR, rr = threadIdx.x / TPR;
  const int64_t chunks = K / 8;
  int par = 0;
  for (int64_t n0 = (int64_t)blockIdx.x * RPC; n0 < N; n0 += (int64_t)gridDim.x * RPC, par ^= 1) {
    const int64_t n = n0 + rr;
    const bool in = n < N;
    const uint4* row = reinterpret_cast<const uint4*>(w + (in ? n : 0) * K);
    uint4 v[kFp8Keep];
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < kFp8Keep; ++i) {
      const int64_t c = rt + (int64_t)i * TPR;
      v[i] = in && c < chunks ? row[c] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < kFp8Keep; ++i) m = absmax8(v[i], m);
    for (int64_t c = rt + (int64_t)kFp8Keep * TPR; in && c < chunks; c += TPR) m = absmax8(row[c], m);
    m = max(m & 0xffffu, m >> 16);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if constexpr (TPR > 32) {
      if (lane == 0) red[par][warp] = m;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < TPR / 32; ++i) m = max(m, red[par][i]);
    }
    float amax = __half2float(__ushort_as_half((uint16_t)m));
    const bool bad = m >= 0x7c00u;  // uniform over the row's threads
    if (bad) {
      // the largest magnitude that is not NaN, as fmaxf takes it
      float a = 0.0f;
      for (int64_t c = rt; in && c < chunks; c += TPR) {
        float f[8];
        halves8(row[c], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) a = fmaxf(a, fabsf(f[e]));
      }
      a = warp_max(a);
      if constexpr (TPR > 32) {
        if (lane == 0) redf[par][warp] = a;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TPR / 32; ++i) a = fmaxf(a, redf[par][i]);
      }
      amax = a;
      if (rt == 0 && in) atomicOr(&g_quant_status, SQ_DEV_NONFINITE_WEIGHT);
    }
    const float s = __fdiv_rn(amax, 448.0f);
    // (-1: under a zero or infinite scale the bounds of a number differ, so those
    // rows take the division's path)
    const float r = s > 0.0f ? __fdiv_rn(1.0f, s) : 0.0f;
    const float rlo = bad || s == 0.0f ? -1.0f : r * (1.0f - 0x1p-21f), rhi = r * (1.0f + 0x1p-21f);
    if (in) {
      if (rt == 0) scales[n] = s;
      uint2* out = reinterpret_cast<uint2*>(codes + n * K);
#pragma unroll
      for (int i = 0; i < kFp8Keep; ++i) {
        const int64_t c = rt + (int64_t)i * TPR;
        if (c < chunks) out[c] = fp8_codes8(v[i], s, rlo, rhi);
      }
      for (int64_t c = rt + (int64_t)kFp8Keep * TPR; c < chunks; c += TPR) out[c] = fp8_codes8(row[c], s, rlo, rhi);
    }
  }
}

cudaError_t launch_quant_int4(const void* w, int64_t N, int64_t K, void* codes, void* scales,
                              cudaStream_t st) {
  const int64_t total = N * (K / 8);
  if (total == 0) return cudaSuccess;
  const int64_t cap = (int64_t)device_sm_count() * 16;
  const bool few = total <= (int64_t)device_sm_count() * 4 * kQuantThreads;
  const int64_t per = (few ? 1 : 4) * kQuantThreads;
  const int64_t want = (total + per - 1) / per;
  return launch_pdl(few ? quant_int4_kernel<1> : quant_int4_kernel<4>, dim3((unsigned)(want < cap ? want : cap)),
                    dim3(kQuantThreads), 0, st,
                    reinterpret_cast<const __half*>(w), N, K, reinterpret_cast<uint8_t*>(codes),
                    reinterpret_cast<__half*>(scales));
}

cudaError_t launch_quant_fp8(const void* w, int64_t N, int64_t K, void* codes, void* scales,
                             cudaStream_t st) {
  if (N == 0) return cudaSuccess;
  // a warp per row while its registers hold the row and there are rows for three
  // warps an SM (100 x 1024: 3.1 us, a CTA per row 2.1; 600 x 1024: 3.2, 3.7;
  // 1000 x 1024: 3.2, 5.0), else a CTA
  const bool one_warp = K <= 32 * 8 * kFp8Keep && N >= (int64_t)device_sm_count() * 3;
  const int rpc = one_warp ? kQuantThreads / 32 : 1;
  const int64_t want = (N + rpc - 1) / rpc, cap = (int64_t)device_sm_count() * 8;
  const dim3 grid((unsigned)(want < cap ? want : cap));
  return launch_pdl(one_warp ? quant_fp8_kernel<32> : quant_fp8_kernel<kQuantThreads>, grid, dim3(kQuantThreads),
                    0, st, reinterpret_cast<const __half*>(w), N, K, reinterpret_cast<uint8_t*>(codes),
                    reinterpret_cast<float*>(scales));
}

cudaError_t take_quant_status(uint32_t* bits) {
  uint32_t v = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_quant_status, sizeof(v));
  if (e != cudaSuccess) return e;
  if (v) e = cudaMemcpyToSymbol(g_quant_status, &zero, sizeof(zero));
  *bits |= v;
  return e;
}

}  // namespace sq
