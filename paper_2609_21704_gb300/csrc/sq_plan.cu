// sq_plan.cu -- how a linear call runs: device properties, the choice of
// engine (streaming, ring, tcgen05 tiles or CUDA-core GEMV, asked in this order)
// and, for the GEMV, the activation-row chunking and the rows-per-group /
// lanes-per-row configuration.  Host code only; the kernels live in
// sq_stream.cu, sq_ring.cu, sq_tc.cu and sq_gemv*.cu, argument checking in
// sq_capi.cu.
#include <stdlib.h>

#include "sq_internal.h"

namespace sq {

int device_sm_count() {
  static int cache[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return kNumSMs;
  if (cache[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
      n = kNumSMs;
    cache[dev] = n;
  }
  return cache[dev];
}

bool pdl_enabled() {
  static const bool on = [] {
    const char* e = getenv("SQ_PDL");
    return !(e && e[0] == '0');
  }();
  return on;
}

int device_max_smem() {
  static int cache[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 227 * 1024;
  if (cache[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        n <= 0)
      n = 227 * 1024;
    cache[dev] = n;
  }
  return cache[dev];
}

// ---------------------------------------------------------------- GEMV plan

static int sub_of(int wk) { return wk == SQ_W_INT4 ? 4 : wk == SQ_W_FP8 ? 2 : 1; }
int64_t weights_per_piece(int wk) { return wk == SQ_W_INT4 ? 32 : wk == SQ_W_FP8 ? 16 : 8; }
int64_t row_bytes_of(int wk, int64_t K) {
  return wk == SQ_W_INT4 ? K / 2 : wk == SQ_W_FP8 ? K : 2 * K;
}

size_t gemv_smem_bytes(int wk, int mr, int64_t K) {
  const int64_t pieces = K / weights_per_piece(wk);
  const int64_t ppad = (pieces + 31) / 32 * 32;
  // staged x, plus one fp32 offset per (row, piece) for INT4
  return (size_t)mr * (size_t)ppad * ((size_t)sub_of(wk) * 16u + (wk == SQ_W_INT4 ? 4u : 0u));
}

// Compiled activation-row counts (sq_gemv.cuh instantiations).
static const int kMRs[] = {1, 2, 4, 5, 8, 16};

int gemv_pick_mr(int M) {
  for (int mr : kMRs)
    if (M <= mr) return mr;
  return 16;
}

// Largest compiled MR whose staged x fits in shared memory.
int gemv_cap_mr(int wk, int64_t K) {
  const size_t limit = (size_t)device_max_smem() - 1024;
  int best = 0;
  for (int mr : kMRs)
    if (gemv_smem_bytes(wk, mr, K) <= limit) best = mr;
  return best;
}

// Tensor cores or CUDA cores, for the calls that neither the streaming engine
// nor the ring takes.  From 16 rows on a CUDA-core GEMV is issue bound (16 fused
// multiply-adds per weight); below that the choice follows timings of both paths
// on the 1.5B/7B/14B projection shapes:
//   * 8..15 rows: tensor cores for FP16 and FP8 weights (1.5-3x faster on
//     every shape), and for INT4 weights from 8 Mi weights on (the INT4
//     GEMV keeps small matrices, where its 8 x dequant reuse still pays);
//   * 3..7 rows, FP16 weights: tensor cores for long rows (K >= 8192), the
//     fused gate/up from 16 Mi weights, and wide outputs (N >= 65536) with
//     K >= 2048; the GEMV for the rest (its many warps fill the GPU better
//     than 128-row tiles do when N is small);
//   * fewer rows, or FP8/INT4 below 8 rows: the GEMV.
bool use_tensor_cores(int wk, int M, int64_t N, int64_t K, int epi) {
  const bool silu = epi == SQ_EPI_SILU_GATE;
  const int64_t weights = (silu ? 2 * N : N) * K;
  if (M >= 16) return true;
  if (M >= 8) return wk != SQ_W_INT4 || weights >= ((int64_t)8 << 20);
  if (wk == SQ_W_FP16 && M >= 3)
    return K >= 8192 || (silu && weights >= ((int64_t)16 << 20)) || (N >= 65536 && K >= 2048);
  return false;
}

cudaError_t launch_gemv(int wk, const GemvArgs& a0, cudaStream_t st) {
  // one INT4 row over many 16-row tiles: products on the tensor cores
  if (gemv_uses_mma(wk, a0.M, a0.N))
    return launch_gemv_mma_int4(a0, a0.epi == SQ_EPI_SILU_GATE, st);
  GemvArgs a = a0;
  const int cap = gemv_cap_mr(wk, a.K);
  if (cap == 0) return cudaErrorInvalidValue;
  // Rows of x are processed in chunks of at most `cap` (each chunk reads the
  // weights once); M <= 16 with K up to ~19k fits in one or two chunks.
  for (int m0 = 0; m0 < a0.M;) {
    const int rem = a0.M - m0;
    int mr = gemv_pick_mr(rem < cap ? rem : cap);
    if (mr > cap) {
      mr = 0;
      for (int c : kMRs)
        if (c <= cap) mr = c;
    }
    const int m_here = rem < mr ? rem : mr;
    a.M = m_here;
    a.x = a0.x + (int64_t)m0 * a0.K;
    a.y = a0.y + (int64_t)m0 * a0.N;
    a.residual = a0.residual ? a0.residual + (int64_t)m0 * a0.N : nullptr;
    const bool silu = a.epi == SQ_EPI_SILU_GATE;
    // rows per lane group and lanes per row, fitted to timings of every
    // projection shape of the 1.5B/7B/14B stacks (within 1 % of the best
    // of the nine (R, LPR) choices overall): two rows per group once there
    // are enough rows to keep every warp busy; SiLU already doubles the
    // rows a group holds
    int r = 1;
    if (mr <= 5) r = (a.N >= 4096 && !silu) ? 2 : 1;
    else r = (mr == 16 && silu) ? 1 : 2;
    // lanes per row: 32 for long rows (>= 256 pieces, several batches per
    // row anyway) and for MR >= 8 (compiled for 32 only); otherwise the
    // largest of 32/16/8 that divides the row's 16-byte pieces (no idle
    // lanes), unless that leaves too few tiles to spread over the warps
    int lpr = 32;
    if (mr <= 5 && a.pieces < 256) {
      for (int cand : {32, 16, 8}) {
        if (a.pieces % cand) continue;
        const int64_t per_tile = (int64_t)(32 / cand) * r;
        const int64_t tiles = (a.N + per_tile - 1) / per_tile;
        if (cand == 32 || tiles >= (int64_t)device_sm_count() * 4) lpr = cand;
        break;
      }
    }
    const int64_t rows_per_tile = (int64_t)(32 / lpr) * r;
    const int64_t ntiles = (a.N + rows_per_tile - 1) / rows_per_tile;
    const int64_t blocks = (ntiles + 7) / 8;
    const size_t smem = gemv_smem_bytes(wk, mr, a.K);
    cudaError_t e;
    if (wk == SQ_W_INT4) e = launch_gemv_int4(a, mr, r, silu, lpr, blocks, smem, st);
    else if (wk == SQ_W_FP8) e = launch_gemv_fp8(a, mr, r, silu, lpr, blocks, smem, st);
    else e = launch_gemv_fp16(a, mr, r, silu, lpr, blocks, smem, st);
    if (e != cudaSuccess) return e;
    m0 += m_here;
  }
  return cudaSuccess;
}

// The shared-memory ring engine (sq_ring.cu), mostly one activation row, where it
// measured faster than the GEMV family (GB300, graphs of whole-stack launch
// sequences; us per launch, ring vs previous engine):
//   INT4 fused gate/up of >= 64 Mi weights (7B, 14B): 14B 19.5 vs 25.8;
//     the 1.5B one (27.5 Mi) stays on the register-operand path (6.9 vs 5.0);
//   FP16 fused gate/up of >= 16 Mi weights: 14B 49.5 vs 54.0, 1.5B 10.0 vs
//     11.3; FP16 lm_head (N >= 65536): 14B 228 vs 375, 1.5B 74.6 vs 79.5;
//   FP8 lm_head of >= 400 Mi weights: 14B 124 vs 164 (1.5B: 46.0 vs 41.1), and at
//     two to eight rows, against the streaming engine, of >= 200 Mi (use_stream).
// q/k/v, o and down (96..448 tiles of 16 rows) stay on the GEMV family: at
// 2-3 tiles per SM the ring's whole-tile work split leaves SMs idle.
bool use_ring(int wkind, int M, int64_t N, int64_t K, int epi) {
  if (!ring_supported(wkind, M, K)) return false;
  const bool silu = epi == SQ_EPI_SILU_GATE;
  const int64_t weights = (silu ? 2 * N : N) * K;
  const int64_t Mi = (int64_t)1 << 20;
  if (M > 1) return wkind == SQ_W_FP8 && !silu && N >= 65536 && weights >= 200 * Mi;
  switch (wkind) {
    case SQ_W_INT4: return silu && weights >= 64 * Mi;
    case SQ_W_FP16: return (silu && weights >= 16 * Mi) || (!silu && N >= 65536);
    case SQ_W_FP8: return !silu && weights >= 400 * Mi;
  }
  return false;
}

// The streaming engine (sq_stream.cu) where it measured faster than the engines
// below: us a launch, weights cold, graphs of the same call with each engine forced
// in turn (139 shapes, 512 .. 152064 outputs, K 1024 .. 18944, plain and gated), and
// whole passes of the 1.5B, 7B and 14B stacks with one projection's engine changed,
// which decide where the two disagree (kernels of different shared-memory needs
// overlap less).
//   INT4, one row: the lm_head of >= 400 Mi weights (14B 80.5 -> 74.2); smaller
//     matrices stay on the GEMV family, whose lanes need no partial sums (1.5B
//     q/k/v 2.4 against 3.3), and the fused gate/up on the ring (alone it gains,
//     but between launches of the GEMV family the four 14B layers take 253 us
//     instead of 196).
//   INT4 and FP8, 2 .. 8 rows: everything (14B q/k/v INT4 at 2 rows 10.6 -> 8.5,
//     down FP8 at 8 rows 36.8 -> 17.2) but the FP8 lm_head of >= 200 Mi, which
//     the ring streams as fast as memory gives (14B at 2 rows 127 against 133).
//   INT4, 9 .. 16 rows: everything, as the other engines spend their time on the
//     conversion (14B lm_head at 16 rows 196 -> 137, 512 x 8192 at 12 rows 22.8 ->
//     7.0); at 16 rows, where the tile path takes small matrices too, from 3 Mi
//     weights on (1536 x 1536 4.4 against 5.2).
//   FP8, 9 .. 16 rows: everything (14B lm_head at 16 rows 272 -> 167) but plain
//     outputs of K >= 2048 in up to 8 weight tiles, whose K the tile path splits over
//     many CTAs (512 x 8192 at 16 rows 6.7 against 9.0), and, from 14 rows on, where
//     the staged rows take most of the shared memory, of 25 to 39 tiles (4096 x 8192
//     13.4 against 15.4; 7B passes at 16 rows with the down projection here 711 us
//     against 686, with q/k/v 699, but 14B's down, 40 tiles, 464 against 476).
//   FP16, plain.  The tile path runs two CTAs an SM up to 76 weight tiles: there
//     it is the faster one for long rows (K >= 8192: 14B down at 5 rows 25.9
//     against 27.6) and at eight rows from K = 2048 on (7B q/k/v 8.4 against 8.9);
//     else the streaming engine is (14B q/k/v at 5 rows 18.9 -> 15.4, 24576 x 1536 at
//     8 rows 21.8 -> 14.7): from 8 Mi weights on, or, at six and seven rows, where the
//     alternative is the GEMV, any (896 x 4864 10.3 -> 6.4).  Its lm_head of >= 400
//     Mi takes two rows only (14B 383 -> 254; at five 251 against 257).
//   FP16, gated: from 16 Mi weights on at two rows (7B pass 829 -> 716; 1.5B, 26 Mi,
//     757 -> 690); small ones at six and seven rows (GEMV: 1024 x 4096 15.0 -> 7.5);
//     short rows below 32 Mi at three to six (1.5B pass at three rows 727 -> 711, at
//     five 753 -> 732; at six 754 against 771 between linear calls alone, but 1610 ->
//     1579 in a decoder pass) and few long rows (512 x 16384 at three 14.1 -> 10.7);
//     the tile path has the rest (7B pass at three rows 636 against 654).
bool use_stream(int wkind, int M, int64_t N, int64_t K, int epi) {
  if (!stream_supported(wkind, M, N, K, epi)) return false;
  const bool silu = epi == SQ_EPI_SILU_GATE;
  const int64_t Mi = (int64_t)1 << 20;
  const int64_t weights = (silu ? 2 * N : N) * K;
  const bool head = !silu && N >= 65536;
  const int64_t tiles = (N + 127) / 128;  // of the tile path
  if (M == 1) return wkind == SQ_W_INT4 && head && weights >= 400 * Mi;
  if (wkind == SQ_W_FP16) {
    if (M > 8) return false;
    if (head) return weights < 400 * Mi ? M >= 3 : M == 2;
    if (silu) {
      if (M == 2) return weights >= 16 * Mi;
      if (weights < 16 * Mi) return M == 6 || M == 7 || (M == 8 && K <= 2048);
      return (M <= 6 && K <= 2048 && weights < 32 * Mi) || tiles <= 8;
    }
    if (M == 2) return false;
    if (M == 8) return K < 2048 || tiles > 76;
    return K >= 8192 ? tiles > 76 : M >= 6 || weights >= 8 * Mi;
  }
  if (M <= 8) return !(wkind == SQ_W_FP8 && head && weights >= 200 * Mi);
  if (wkind == SQ_W_INT4) return M < 16 || weights >= 3 * Mi;
  return silu || K < 2048 || (tiles > 8 && (M < 14 || tiles <= 24 || tiles >= 40));
}

}  // namespace sq
