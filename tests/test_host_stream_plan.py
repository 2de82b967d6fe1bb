"""The streaming engine's host arithmetic (csrc/sq_stream_plan.h), compiled for
the CPU and checked over sizes and cluster counts: a kernel never gets a split
with which its loops stand still, every part of K holds a unit in every CTA of a
cluster, the layout stays inside the shared memory (above half of it where a call
streams much), and the estimate by which a
split is chosen covers all of its passes."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHECK = r"""
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include <vector>
#include "sq_stream_plan.h"
using namespace sq;

static void die(const char* what, int wk, bool silu, const StreamPlan& a, int clusters) {
  std::printf("%s: kind %d silu %d M %d N %lld K %d KS %d clusters %d: S %d pass_tiles %d\n", what, wk, (int)silu,
              a.M, (long long)a.N, a.K, a.KS, clusters, a.S, a.pass_tiles);
  std::exit(1);
}

// Every (tile, part) of a CTA with `rows` rows and `nu` units: taken once, by one
// warp, and copied in the order in which it is multiplied.  The copies of a warp
// are a sequence of jobs that goes on only while the current one has units left.
static bool walk(const StreamPlan& a, int nw, int rows, int nu) {
  const int ntiles = (rows + 15) / 16;
  std::vector<char> taken((size_t)ntiles * a.S, 0);
  for (int warp = 0; warp < nw; ++warp) {
    int it0 = 0, ijj = warp;
    for (int t0 = 0; t0 < ntiles; t0 += a.pass_tiles) {
      const int nt = ntiles - t0 < a.pass_tiles ? ntiles - t0 : a.pass_tiles;
      for (int jj = warp; jj < nt * a.S; jj += nw) {
        const int tile = t0 + jj / a.S, part = jj % a.S;
        while (it0 < ntiles && ijj >= (ntiles - it0 < a.pass_tiles ? ntiles - it0 : a.pass_tiles) * a.S) {
          it0 += a.pass_tiles;
          ijj = warp;
        }
        if (it0 + ijj / a.S != tile || ijj % a.S != part) return false;
        if ((part + 1) * nu / a.S - part * nu / a.S < 1) return false;
        ijj += nw;
        if (taken[(size_t)tile * a.S + part]++) return false;
      }
    }
  }
  for (char c : taken)
    if (!c) return false;
  return true;
}

static long plans = 0;
static void check(int wk, bool silu, int M, int64_t N, int K, int ks, int clusters) {
  if (!s_fits(wk, M, K, ks) || clusters > N) return;
  const int nw = s_warps(M == 1 ? 0 : M <= 8 ? 1 : 2);
  StreamPlan a = {};
  a.M = M;
  a.K = K;
  a.N = N;
  a.row_bytes = wk == SQ_W_INT4 ? K / 2 : wk == SQ_W_FP8 ? K : 2 * (int64_t)K;
  a.U = s_units(wk, K);
  a.KS = ks;
  double ns = -1.0;
  const int smem = s_split(wk, silu, nw, clusters, a, &ns);
  ++plans;
  // what fits gets a split (no call that the rule sends here is refused)
  if (smem <= 0 || !(ns > 0.0)) die("no split", wk, silu, a, clusters);
  // the loops over passes advance
  if (a.pass_tiles < 1 || a.S < 1) die("a pass without tiles", wk, silu, a, clusters);
  const int64_t tiles = ((N + clusters - 1) / clusters + 15) / 16;
  // the CTAs of a cluster hold floor or ceil(U / KS) units
  if (a.S > a.U / a.KS) die("a part without units", wk, silu, a, clusters);
  if (plans % 61 == 0)
    for (int up = 0; up < 2; ++up)
      if (!walk(a, nw, (int)((N + up * (clusters - 1)) / clusters), (a.U + up * (ks - 1)) / ks))
        die("jobs", wk, silu, a, clusters);
  // the estimate counts every round of the warps, those of all passes
  long rounds = 0;
  for (int64_t t = 0; t < tiles; t += a.pass_tiles)
    rounds += ((tiles - t < a.pass_tiles ? tiles - t : a.pass_tiles) * a.S + nw - 1) / nw;
  const int nu = (a.U + ks - 1) / ks;
  if (ns < 330.0 * (silu ? 2 : 1) * rounds * ((nu + a.S - 1) / a.S)) die("rounds not counted", wk, silu, a, clusters);
  const bool direct = a.S == 1 && a.KS == 1;
  const int bufs = direct ? 0 : a.pass_tiles < tiles ? 2 : 1;
  if (!direct && (int64_t)a.pass_tiles * a.S * (silu ? 2 : 1) * 16 * M > a.red_floats)
    die("partial sums past their buffer", wk, silu, a, clusters);
  if (a.off_red + (int64_t)bufs * a.red_floats * 4 > a.off_ring) die("overlap", wk, silu, a, clusters);
  if (a.ns < 3 || a.off_ring + a.ns * nw * kSlotBytes > smem || smem > kSmemMax) die("shared memory", wk, silu, a, clusters);
  // with much to stream no second CTA shares the SM
  if ((N + clusters - 1) / clusters * (silu ? 2 : 1) * a.row_bytes / ks > 96 * 1024 && smem <= kSmemHalf)
    die("two CTAs an SM", wk, silu, a, clusters);
}

int main() {
  // clusters of 1, 2, 4, 8 CTAs that can be resident: full GPUs and fragments of one
  const int counts[4][4] = {{152, 148, 132, 1}, {76, 72, 66, 1}, {38, 36, 30, 1}, {19, 16, 15, 1}};
  const int kinds[3] = {SQ_W_INT4, SQ_W_FP8, SQ_W_FP16}, ku[3] = {128, 64, 32};
  // sizes whose rounding to whole rounds of the warps once gave passes of no tile
  for (int c = 0; c < 4; ++c)
    for (int j = 0; j < 4; ++j) {
      for (int64_t N : {24321, 25699, 26752}) {
        check(SQ_W_FP16, false, 8, N, 8224, 1 << c, counts[c][j]);
        check(SQ_W_FP8, true, 4, N, 16448, 1 << c, counts[c][j]);
      }
      check(SQ_W_FP8, false, 3, 12355, 49216, 1 << c, counts[c][j]);
    }
  for (int k = 0; k < 3; ++k)
    for (int M = 1; M <= 16; ++M)
      for (int U = 1; U <= 2048; U += U < 300 ? 1 : 1 + U / 37)
        for (int c = 0; c < 4; ++c)
          for (int n : counts[c])
            for (int silu = 0; silu < 2; ++silu)
              for (int t = 1; t <= 1200; t += t < 48 ? 1 : t / 4)
                check(kinds[k], silu, M, (int64_t)n * 16 * t - (U + t) % (16 * n), U * ku[k], 1 << c, n);
  std::printf("%ld plans\n", plans);
  return 0;
}
"""


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    d = tmp_path_factory.mktemp("stream_plan")
    (d / "check.cpp").write_text(CHECK)
    exe = str(d / "check")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2609_21704_gb300", "csrc"), str(d / "check.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def test_every_split_makes_progress_and_fits(checker):
    r = subprocess.run([checker], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[0]) > 1_000_000
