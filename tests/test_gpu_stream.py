"""GPU parity of the streaming engine against the fp64 oracle over the same
dequantised weights: fewer output rows than SMs, ragged tiles, one unit of K and
odd unit counts, the row counts at which its column tiles change (2, 8, 9, 16),
K split over a cluster with one and with several passes of partial sums, the
epilogues, the fused RMSNorm, non-finite activations, and the precision of INT4 sums.
Bar: relative L2 <= 1e-3, max-abs <= 2e-2."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_21704_gb300 as sq
from paper_2609_21704_gb300 import synth

from gpu_util import assert_close, bits16, dev, dev_to_f64, f16_to_dev

pytestmark = pytest.mark.gpu

WK = {"int4": sq.SQ_W_INT4, "fp8": sq.SQ_W_FP8, "fp16": sq.SQ_W_FP16}
NONE, SILU, RES = sq.SQ_EPI_NONE, sq.SQ_EPI_SILU_GATE, sq.SQ_EPI_RESIDUAL


def _weights(kind, rows, K, seed):
    """Device weight, scales, and fp64 rows (by index) of a seeded matrix."""
    w16 = synth.weights_fp16_device(seed, rows, K, dev())
    if kind == "fp16":
        return w16, None, lambda i: bits16(w16[i]).view(np.float16).astype(np.float64)
    qk = sq.SQ_INT4_G128 if kind == "int4" else sq.SQ_FP8_E4M3_ROW
    cb, _ = sq.sq_quantized_bytes(qk, rows, K)
    codes = torch.empty(rows, cb // rows, dtype=torch.uint8, device=dev())
    scales = torch.empty((rows, K // 128) if kind == "int4" else (rows,),
                         dtype=torch.float16 if kind == "int4" else torch.float32, device=dev())
    sq.sq_quantize(w16, qk, codes, scales)

    def rows64(i):
        b = bits16(w16[i])
        return oracle.dequant_int4(*oracle.quantize_int4(b), K) if kind == "int4" else \
            oracle.dequant_fp8(*oracle.quantize_fp8(b))
    return codes, scales, rows64


def _call(kind, M, N, K, epi=NONE, seed=0, x=None, norm=False):
    assert sq.sq_linear_path(WK[kind], M, N, K, epi) == 4
    rows = 2 * N if epi == SILU else N
    w, s, rows64 = _weights(kind, rows, K, seed + N + K)
    if x is None:
        x = synth.activations_fp16(seed + 5 * M + K, M, K)
    xt = f16_to_dev(x)
    bias = synth.fp16_normal(seed + 3, (rows,), 0.5)
    res = synth.activations_fp16(seed + 9, M, N) if epi == RES else None
    y = torch.full((M, N), 9.0, dtype=torch.float16, device=dev())
    rt = f16_to_dev(res) if res is not None else None
    x64 = x.astype(np.float64)
    if norm:
        g = (1 + synth.fp16_normal(seed + 4, (K,), 0.1).astype(np.float32)).astype(np.float16)
        xn = torch.empty(M, K, dtype=torch.float16, device=dev())
        sq.sq_linear_norm(WK[kind], xt, f16_to_dev(g), 1e-6, xn, w, s, f16_to_dev(bias), rt, epi, y)
        x64 = oracle.rmsnorm(x64, g.astype(np.float64), 1e-6)
        y2 = torch.empty_like(y)
        sq.sq_rmsnorm(xt, f16_to_dev(g), 1e-6, xn)
        sq.sq_linear_ex(WK[kind], xn, w, s, f16_to_dev(bias), rt, epi, y2)
        assert torch.equal(y.view(torch.int16), y2.view(torch.int16)), "not the two calls' bits"
    else:
        sq.sq_linear_ex(WK[kind], xt, w, s, f16_to_dev(bias), rt, epi, y)
    assert sq.sq_check() == 0
    cols = np.arange(N) if N <= 600 else np.unique(np.append(np.random.default_rng(N).integers(0, N, 500), [0, N - 1]))
    idx = torch.from_numpy(np.concatenate([cols, cols + N]) if epi == SILU else cols).to(dev())
    with np.errstate(invalid="ignore"):
        ref = x64 @ rows64(idx).T + bias[idx.cpu().numpy()].astype(np.float64)[None, :]
    if epi == SILU:
        ref = oracle.silu_gate(ref[:, :len(cols)], ref[:, len(cols):])
    if epi == RES:
        ref = ref + res[:, cols].astype(np.float64)
    return dev_to_f64(y)[:, cols], ref


CASES = [
    # kind, M, N, K, epi
    ("int4", 2, 1, 128, NONE), ("int4", 8, 17, 128, RES), ("int4", 9, 151, 384, NONE), ("int4", 5, 2433, 896, SILU),
    ("int4", 16, 4000, 1536, SILU), ("int4", 16, 2500, 8960, RES), ("int4", 12, 30000, 5120, NONE),
    ("int4", 1, 82000, 5120, NONE), ("int4", 3, 200, 18944, NONE),
    ("fp8", 2, 3, 64, NONE), ("fp8", 8, 2431, 192, RES), ("fp8", 9, 153, 1088, SILU), ("fp8", 16, 20000, 5120, NONE),
    ("fp8", 11, 3584, 18944, NONE), ("fp8", 16, 3000, 2048, SILU),
    ("fp16", 2, 9000, 4096, SILU), ("fp16", 5, 5120, 5120, RES), ("fp16", 3, 9800, 8224, RES),
    ("fp16", 7, 1543, 1568, NONE), ("fp16", 6, 70001, 1536, NONE),
    # ragged last tiles, long rows and large outputs, few rows and many
    ("int4", 2, 7168 + 5, 5120, NONE), ("int4", 3, 1000, 2048, RES), ("int4", 4, 13824, 5120, SILU),
    ("int4", 5, 5120, 5120, NONE), ("int4", 8, 4133, 1536, SILU), ("int4", 8, 152064, 5120, NONE),
    ("int4", 4, 5120, 13824, RES), ("int4", 2, 3000, 27648, SILU), ("int4", 8, 1003, 8192, RES),
    ("int4", 9, 1024, 8192, NONE), ("int4", 13, 2048, 4096, NONE), ("int4", 16, 8192, 5120, NONE),
    ("int4", 16, 6912, 5120, SILU), ("fp8", 8, 7168, 5120, NONE), ("fp8", 5, 300, 1024, SILU),
    ("fp8", 4, 37, 13824, RES), ("fp8", 16, 16384, 4096, SILU),
    ("fp16", 8, 24321, 8224, NONE),  # thirteen parts for twelve warps were once the cheapest split: no whole round
]


@pytest.mark.parametrize("kind,M,N,K,epi", CASES)
def test_matches_oracle(kind, M, N, K, epi):
    assert_close(*_call(kind, M, N, K, epi), f"{kind} M={M} N={N} K={K} epi={epi}")


@pytest.mark.parametrize("kind,M,N,K", [("int4", 2, 500, 1536), ("int4", 16, 700, 5120), ("fp8", 7, 300, 1024),
                                        ("fp16", 8, 400, 1536)])
def test_fused_norm(kind, M, N, K):
    assert_close(*_call(kind, M, N, K, norm=True, seed=3), f"{kind} norm M={M}")


@pytest.mark.parametrize("kind", ["int4", "fp8"])
@pytest.mark.parametrize("M,N,K", [(2, 300, 1024), (16, 2500, 5120)])
def test_nonfinite_activations_stay_in_their_row(kind, M, N, K):
    x = synth.activations_fp16(8, M, K)
    x[0, 77] = np.float16(np.inf)
    x[M - 1, K - 3] = np.float16(-np.inf)
    x[M - 1, 5] = np.float16(np.inf)
    if M > 2:
        x[1, 9] = np.float16(np.nan)
    got, ref = _call(kind, M, N, K, x=x)
    fin = [m for m in range(M) if np.all(np.isfinite(x[m]))]
    if fin:
        assert_close(got[fin], ref[fin], "finite rows")
    # an infinity times a code of zero is NaN, like in the definition
    for m in set(range(M)) - set(fin):
        assert np.array_equal(np.isnan(got[m]), np.isnan(ref[m])), m
        ok = ~np.isnan(ref[m])
        assert np.array_equal(got[m][ok], ref[m][ok]), m


@pytest.mark.parametrize("M,N,K", [(1, 82000, 5120), (2, 1536, 8960), (8, 4608, 3584), (16, 4000, 1536)])
def test_int4_sums_keep_fp32_precision(M, N, K):
    """Activations as the gate leaves them: their products with exact codes, in fp32
    sums, seldom move an fp16 result.  A sum of about a hundred rounded group sums of
    up to its own size is off by some 10 * 2^-24 of the row's RMS, so about 1 in 1000
    results (an fp16 step is 2^-10 of the largest) rounds the other way; sums that
    drop the seven lowest bits turn 2 in 100 and more."""
    rng = np.random.default_rng(M + K)
    g, u = rng.normal(size=(2, M, K))
    x = (g / (1 + np.exp(-g)) * np.abs(u)).astype(np.float16)
    w, s, rows64 = _weights("int4", N, K, 3 * N + K)
    y = torch.empty(M, N, dtype=torch.float16, device=dev())
    sq.sq_linear_ex(sq.SQ_W_INT4, f16_to_dev(x), w, s, None, None, NONE, y)
    assert sq.sq_check() == 0
    cols = np.unique(rng.integers(0, N, 4000 // M + 200))
    ref = x.astype(np.float64) @ rows64(torch.from_numpy(cols).to(dev())).T
    wrong = np.mean(dev_to_f64(y)[:, cols] != ref.astype(np.float16).astype(np.float64))
    assert wrong < 0.006, wrong
