"""sq_quantize, bit exact against the oracle, where its kernels change path:
partial warps of INT4 groups, FP8 rows around what a warp's and a CTA's
registers hold, quotients on and next to a rounding tie, scales at the
bottom of the fp16 range (codes by division), and rows without a finite maximum."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_21704_gb300 as sq
from paper_2609_21704_gb300 import synth

from gpu_util import bits16, dev, f16_to_dev

pytestmark = pytest.mark.gpu


def _check(w, kind):
    N, K = w.shape
    cb, _ = sq.sq_quantized_bytes(kind, N, K)
    codes = torch.empty(cb, dtype=torch.uint8, device=dev())
    i4 = kind == sq.SQ_INT4_G128
    scales = torch.empty(N * (K // 128) if i4 else N, dtype=torch.float16 if i4 else torch.float32, device=dev())
    sq.sq_quantize(f16_to_dev(w), kind, codes, scales)
    assert sq.sq_check() == 0
    oc, os_ = (oracle.quantize_int4 if i4 else oracle.quantize_fp8)(w.view(np.uint16))
    assert np.array_equal(codes.cpu().numpy().reshape(N, -1), oc)
    if i4:
        assert np.array_equal(bits16(scales).reshape(N, -1), os_)
    else:
        assert np.array_equal(scales.cpu().numpy().view(np.uint32), os_.view(np.uint32))


def _rows(N, K, seed):
    """Weights of all magnitudes, many of them a half-integer multiple of the
    scale their group gets (amax 7 x 2^e, 3.5 x 2^e), and signed zeros."""
    rng = np.random.default_rng(seed)
    w = synth.weights_fp16(seed, N, K).copy()
    for n in range(N):
        e = int(rng.integers(-24, 12))
        if n % 3 == 0:
            w[n] = (rng.integers(-14, 15, K) * 0.5 * 2.0 ** e).astype(np.float16)
            w[n, ::64] = np.float16(min(7.0 * 2.0 ** e, 60000.0))
        elif n % 3 == 1:
            w[n] = (w[n].astype(np.float64) * 2.0 ** e).astype(np.float16)
    w[N // 2] = np.float16(-0.0)
    return w


@pytest.mark.parametrize("N,K", [(1, 128), (3, 384), (9, 128), (37, 1152), (130, 256),
                                 (1216, 1024), (1217, 1024)])  # the most with 256 weights a warp, the least with 1024
def test_int4_partial_warps_ties_and_small_scales(N, K):
    _check(_rows(N, K, N + K), sq.SQ_INT4_G128)


@pytest.mark.parametrize("N,K", [(5, 2032), (9, 2048), (5, 2064), (2, 16384), (3, 16400), (2, 40000),
                                 (455, 272), (456, 272), (459, 2032), (461, 2048), (460, 2064)])  # a warp per row
def test_fp8_row_lengths_ties_and_small_scales(N, K):
    _check(_rows(N, K, N + K), sq.SQ_FP8_E4M3_ROW)


@pytest.mark.parametrize("N", [4, 460])  # a CTA per row, a warp per row
@pytest.mark.parametrize("K", [16, 2048, 4112])
def test_fp8_rows_of_nan_and_zeros_get_code_zero(N, K):
    """A row whose largest number is zero has scale 0 and codes +0, also where
    eight neighbouring weights are all NaN (both bounds of a quotient are)."""
    w = np.zeros((N, K), dtype=np.float16)
    w[0] = np.nan
    w[1, 8:16] = np.nan
    w[2, K - 8:K - 1] = np.nan
    w[3] = -0.0
    codes = torch.full((N, K), 7, dtype=torch.uint8, device=dev())
    scales = torch.full((N,), 7.0, dtype=torch.float32, device=dev())
    sq.sq_quantize(f16_to_dev(w), sq.SQ_FP8_E4M3_ROW, codes, scales)
    assert sq.sq_check() & sq.SQ_DEV_NONFINITE_WEIGHT
    assert not scales.any()
    assert not codes.any()
