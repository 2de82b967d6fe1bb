// sq_stream_plan.h -- host arithmetic of the streaming engine (sq_stream.cu): how
// a call is split over clusters, warps and passes, and its shared-memory layout.
// No CUDA, so that it can be checked over all sizes without a GPU.
#pragma once

#include <stdint.h>

#include "specquant.h"

namespace sq {

// NT: 0 one activation row, 1 up to eight (one column tile), 2 up to sixteen.
// Warps of a CTA: twelve; sixteen (and so one CTA per SM) for one row, the
// lm_head, whose many long rows want warps more than a neighbour (14B INT4: 72
// us against 80).
constexpr int s_warps(int nt) { return nt == 0 ? 16 : 12; }
constexpr int kSmemMax = 227 * 1024;
constexpr int kSmemHalf = 113 * 1024;
constexpr int kSlotBytes = 2048;  // one warp's step: [2][row g, row g + 8][lane] 16-byte pieces
constexpr int kMaxRows = 16;

struct StreamPlan {
  int M;
  int K;
  int64_t N, row_bytes;
  int U;            // 64-byte units of a weight row
  int KS;           // CTAs of a cluster along K
  int S;            // parts of a CTA's units, one job each
  int pass_tiles;   // tiles whose partial sums meet at once
  int xstride;      // shared bytes between staged rows
  int off_misc;     // RMSNorm scratch
  int off_red;      // one or two buffers of partial sums
  int red_floats;   // floats of one buffer
  int off_ring;
  int ns;           // ring slots per warp, 3 or 4
};

inline int s_units(int wkind, int64_t K) { return (int)(K / (wkind == SQ_W_INT4 ? 128 : wkind == SQ_W_FP8 ? 64 : 32)); }

// Shared memory up to the partial sums: staged rows, RMSNorm scratch.
inline int s_fixed(int wkind, int M, int nu, StreamPlan& a) {
  const int ku = wkind == SQ_W_INT4 ? 128 : wkind == SQ_W_FP8 ? 64 : 32;
  a.xstride = (nu * ku * 2 + 127) / 128 * 128 + 64;
  a.off_misc = (M * a.xstride + 127) / 128 * 128;
  a.off_red = a.off_misc + (kMaxRows + 8 * kMaxRows) * 4;
  return a.off_red;
}

// Does the call fit with K split over ks CTAs (ring, staged rows and 8 KB of
// partial sums)?
inline bool s_fits(int wkind, int M, int64_t K, int ks) {
  const int ku = wkind == SQ_W_INT4 ? 128 : wkind == SQ_W_FP8 ? 64 : 32;
  if (M < 1 || M > kMaxRows || K % ku != 0) return false;
  const int U = s_units(wkind, K), nw = s_warps(M == 1 ? 0 : M <= 8 ? 1 : 2);
  StreamPlan a = {};
  return ks <= U &&
         s_fixed(wkind, M, (U + ks - 1) / ks, a) + 8 * 1024 + 128 + 3 * nw * kSlotBytes <= kSmemMax;
}

// The work split of a call with K over a.KS CTAs and `clusters` clusters: fills
// in S, pass_tiles, the layout and the slots; returns the shared memory and an
// estimate of the time in ns (relative choices only), smem 0 when nothing fits.
inline int s_split(int wkind, bool silu, int nw, int clusters, StreamPlan& a, double* ns) {
  const int wr = silu ? 2 : 1;
  const int nu = (a.U + a.KS - 1) / a.KS;
  const int fixed = s_fixed(wkind, a.M, nu, a);
  const int64_t rows = (a.N + clusters - 1) / clusters;
  const int64_t tiles = (rows + 15) / 16;
  if (rows > (1 << 24)) return 0;
  // Parts of K: the busiest warp's units, one and a half of overhead a job, over
  // the passes that the partial sums need (two buffers where one does not hold
  // them all).  At most one part a warp, so that whole rounds of the warps keep at
  // least a tile a pass: a pass of no tile would never end.  At most one part a
  // unit of the CTA with the fewest: a warp's copies would stop for good at a
  // part without units.  (Costed as if all tiles met at once, 16 rows of an FP8
  // gate/up, 16384 x 4096, took seven passes of five busy warps, 53 us; now four
  // CTAs along K, one pass, 37.)
  const int room = kSmemMax - fixed - 128 - 3 * nw * kSlotBytes;
  double best = -1.0;
  int64_t pt = 0;
  int nbuf = 0;
  for (int S = 1; S <= a.U / a.KS && S <= nw; ++S) {
    const bool direct = S == 1 && a.KS == 1;
    const int per_tile = S * wr * 16 * a.M * 4;
    int64_t p = tiles;
    if (!direct && p * per_tile > room) {
      p = room / 2 / per_tile;
      if (p * S > nw) p = p * S / nw * nw / S;  // whole rounds of the warps
      if (p < 1) break;
    }
    const int64_t full = tiles / p, rest = tiles - full * p;
    const double rounds = (double)(full * ((p * S + nw - 1) / nw) + (rest * S + nw - 1) / nw);
    const double cost = rounds * ((nu + S - 1) / S + 1.5);
    if (best < 0.0 || cost < best) {
      best = cost;
      a.S = S;
      pt = p;
      nbuf = direct ? 0 : p < tiles ? 2 : 1;
    }
    if (tiles >= 4 * nw) break;  // enough whole rows for every warp: no partial sums
  }
  if (pt < 1) return 0;
  a.pass_tiles = (int)pt;
  a.red_floats = nbuf ? (int)pt * a.S * wr * 16 * a.M : 0;
  a.off_ring = (fixed + nbuf * a.red_floats * 4 + 127) / 128 * 128;
  // ring slots: four; a CTA with little to stream rather leaves half the SM's
  // shared memory to the next launch's CTA, which starts its own copies early
  // (1.5B q/k/v at five rows, FP8: 3.4 us against 3.8; with much to stream three
  // slots lose: 14B lm_head at two rows, FP8: 140 us against 132)
  const bool little = rows * wr * a.row_bytes / a.KS <= 96 * 1024;
  a.ns = 4;
  if (a.off_ring + 4 * nw * kSlotBytes > (little ? kSmemHalf : kSmemMax)) a.ns = 3;
  // Estimate, fitted to K splits of 1, 2, 4 and 8 over the 1.5B, 7B and 14B
  // projections at 8, 12 and 16 rows: 330 ns for a unit of every warp, 25 bytes
  // of activations a nanosecond (every CTA reads the same lines), a cluster's
  // launch and its two barriers, one more for every further pass.
  static const double kCluster[9] = {0, 0, 1500, 0, 2500, 0, 0, 0, 6000};
  *ns = best * wr * 330.0 * (a.KS > 1 ? 1.1 : a.ns == 3 && !little ? 1.15 : 1.0) +
        2.0 * a.M * a.K / a.KS / 25.0 + kCluster[a.KS] +
        (a.KS > 1 ? 2000.0 * (double)((tiles + pt - 1) / pt - 1) : 0.0);
  // A call with much to stream takes more than half: another CTA on its SM would
  // slow the one that the call ends with (1.5B FP16 at three rows, whose gate/up
  // just fits in half: a pass of 28 layers and lm_head 830 us, so 797).
  const int smem = a.off_ring + a.ns * nw * kSlotBytes;
  return !little && smem <= kSmemHalf ? kSmemHalf + 1024 : smem;
}

}  // namespace sq
