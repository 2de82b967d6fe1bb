"""GPU parity of the tensor-tile engine where K is split over a cluster and each
rank finishes a share of the output columns: row counts that the split does not
divide, fewer rows than ranks, one and two accumulators, a ragged last weight
tile, every epilogue.  Bar: relative L2 <= 1e-3, max-abs <= 2e-2 (fp32 sums of
fp16 products and one fp16 rounding)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_21704_gb300 as sq
from paper_2609_21704_gb300 import synth

from gpu_util import MAX_ABS, REL_L2, assert_close, dev, dev_to_f64, f16_to_dev, rel_l2

pytestmark = pytest.mark.gpu

WK = {"fp16": sq.SQ_W_FP16, "int4": sq.SQ_W_INT4, "fp8": sq.SQ_W_FP8}


def _weights(kind, w):
    if kind == "fp16":
        return f16_to_dev(w), None, w.astype(np.float64)
    if kind == "int4":
        c, s = oracle.quantize_int4(w.view(np.uint16))
        return torch.from_numpy(c).to(dev()), f16_to_dev(s.view(np.float16)), oracle.dequant_int4(c, s, w.shape[1])
    c, s = oracle.quantize_fp8(w.view(np.uint16))
    return torch.from_numpy(c).to(dev()), torch.from_numpy(s).to(dev()), oracle.dequant_fp8(c, s)


@pytest.mark.parametrize("kind", ["fp16", "int4", "fp8"])
@pytest.mark.parametrize("epi", [sq.SQ_EPI_SILU_GATE, sq.SQ_EPI_RESIDUAL])
@pytest.mark.parametrize("M", [9, 15, 17, 31, 64, 65, 127, 131, 255])
def test_column_shares_match_oracle(kind, epi, M):
    N, K = 200, 4480
    silu = epi == sq.SQ_EPI_SILU_GATE
    rows = 2 * N if silu else N
    w = synth.weights_fp16(M + K, rows, K)
    x = synth.activations_fp16(3 * M + K, M, K)
    b = synth.fp16_normal(M + 7, (rows,), 0.5)
    r = None if silu else synth.fp16_normal(M + 11, (M, N), 1.0)
    wd, sd, w64 = _weights(kind, w)
    y = torch.full((M, N), 9.0, dtype=torch.float16, device=dev())
    sq.sq_linear_ex(WK[kind], f16_to_dev(x), wd, sd, f16_to_dev(b), None if silu else f16_to_dev(r), epi, y)
    assert sq.sq_check() == 0
    full = oracle.linear(x.astype(np.float64), w64, b.astype(np.float64))
    ref = oracle.silu_gate(full[:, :N], full[:, N:]) if silu else full + r.astype(np.float64)
    assert_close(dev_to_f64(y), ref, f"{kind} M={M} epi={epi}")


# two CTAs per SM above 64 rows: both sides of its row and tile limits
@pytest.mark.parametrize("M,N", [(65, 3000), (96, 3072), (97, 3072), (80, 5000), (128, 5120), (129, 5120), (80, 9800)])
def test_two_per_sm_limits_match_oracle(M, N):
    K = 1032
    w = synth.weights_fp16(M + N, N, K)
    x = synth.activations_fp16(M + 2 * N, M, K)
    b = synth.fp16_normal(M + 5, (N,), 0.5)
    y = torch.full((M, N), 9.0, dtype=torch.float16, device=dev())
    sq.sq_linear_ex(sq.SQ_W_FP16, f16_to_dev(x), f16_to_dev(w), None, f16_to_dev(b), None, sq.SQ_EPI_NONE, y)
    assert sq.sq_check() == 0
    ref = oracle.linear(x.astype(np.float64), w.astype(np.float64), b.astype(np.float64))
    assert_close(dev_to_f64(y), ref, f"M={M} N={N}")


# two column blocks: the first and last row counts, K and tile limits, epilogues
@pytest.mark.parametrize("epi", [sq.SQ_EPI_NONE, sq.SQ_EPI_SILU_GATE, sq.SQ_EPI_RESIDUAL])
@pytest.mark.parametrize("M,N,K", [(97, 200, 1536), (128, 1000, 2048), (129, 200, 2056), (161, 130, 1000),
                                   (255, 8960, 72), (256, 9800, 64), (256, 1536, 1536)])
def test_column_blocks_match_oracle(epi, M, N, K):
    silu = epi == sq.SQ_EPI_SILU_GATE
    rows = 2 * N if silu else N
    w = synth.weights_fp16(M + N + K, rows, K)
    x = synth.activations_fp16(M + 2 * K, M, K)
    b = synth.fp16_normal(M + 5, (rows,), 0.5)
    r = synth.fp16_normal(M + 11, (M, N), 1.0) if epi == sq.SQ_EPI_RESIDUAL else None
    y = f16_to_dev(r) if r is not None else torch.full((M, N), 9.0, dtype=torch.float16, device=dev())
    sq.sq_linear_ex(sq.SQ_W_FP16, f16_to_dev(x), f16_to_dev(w), None, f16_to_dev(b), y if r is not None else None,
                    epi, y)
    assert sq.sq_check() == 0
    full = oracle.linear(x.astype(np.float64), w.astype(np.float64), b.astype(np.float64))
    ref = oracle.silu_gate(full[:, :N], full[:, N:]) if silu else full
    if r is not None:
        ref = ref + r.astype(np.float64)
    # gated values reach 90 at K = 1536, where rounding the exact result to fp16
    # alone errs by 2^-11 |ref| = 0.044 (0.0246 seen, on the CPU too): that
    # rounding is allowed per element beside the bound on the sums
    got = dev_to_f64(y)
    assert rel_l2(got, ref) <= REL_L2
    assert np.all(np.abs(got - ref) <= MAX_ABS + 2.0 ** -11 * np.abs(ref)), f"M={M} N={N} K={K} epi={epi}"


def _us(op, copies):
    """Time of one launch: the same call over `copies` weight copies (more than
    the L2 holds) in a graph, best of several replays."""
    st = torch.cuda.Stream()
    ops = [op(i) for i in range(copies)]
    with torch.cuda.stream(st):
        sq.sq_linear_chain(ops, st)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sq.sq_linear_chain(ops, st)
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(st)
            g.replay()
            b.record(st)
            b.synchronize()
            best = min(best, a.elapsed_time(b))
    return 1e3 * best / copies


@pytest.mark.parametrize("tiles,more", [(14, 15), (14, 16), (58, 60)])
def test_split_clusters_run_in_one_wave(tiles, more):
    """A few more weight tiles cost their bytes, not a second wave of the clusters
    (which cost 1.45 to 1.6 times the time; the bytes are at most 1.15)."""
    M, K = 16, 8192
    x = f16_to_dev(synth.activations_fp16(3, M, K))

    def us(t):
        w = [synth.weights_fp16_device(5 + t, 2 * 128 * t, K, dev())]
        copies = max(3, int(3e8 // (4 * 128 * t * K)))
        w += [w[0].clone() for _ in range(copies - 1)]
        y = torch.empty(M, 128 * t, dtype=torch.float16, device=dev())
        return _us(lambda i: (sq.SQ_W_FP16, x, w[i], None, None, None, sq.SQ_EPI_SILU_GATE, y), copies)

    assert us(more) < 1.3 * us(tiles)
