"""GPU parity of the attention kernel's instances against the fp64 oracle: the
query counts at which the launch changes its warp layout (8, 16, 32 and 64
queries per key/value head, and one more), contexts at the edges of a 64-key
block, shares that meet in a cluster and shares that meet in the workspace,
and operands far from 1.  Bar: relative L2 <= 1e-3, max-abs <= 2e-2."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_21704_gb300 as sq

from gpu_util import assert_close, dev

pytestmark = pytest.mark.gpu
D, THETA = 128, 1e6


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dev())


def _case(B, T, Hq, Hkv, pos0, max_ctx, qstd=1.0, fused=False, seed=0):
    rng = np.random.default_rng(seed + 1000 * T + Hq)
    qkv = rng.normal(0, 1, (B * T, (Hq + 2 * Hkv) * D))
    qkv[:, :Hq * D] *= qstd
    qkv = qkv.astype(np.float16)
    g = torch.Generator(device=dev())
    g.manual_seed(seed + 1)
    kc = torch.empty(B, Hkv, max_ctx, D, dtype=torch.float16, device=dev()).normal_(0, 1, generator=g)
    vc = torch.empty_like(kc).normal_(0, 1, generator=g)
    # what lies past the last new token is never read
    for b in range(B):
        kc[b, :, pos0[b] + T:] = float("nan")
        vc[b, :, pos0[b] + T:] = float("inf")
    p0, x = _t(np.array(pos0, np.int32)), _t(qkv)
    out = torch.full((B * T, Hq * D), 7.0, dtype=torch.float16, device=dev())
    ws = torch.empty(sq.sq_attention_workspace_bytes(B, T, Hq, Hkv, max_ctx), dtype=torch.uint8, device=dev())
    if fused:
        sq.sq_attention_append(x, B, T, Hq, Hkv, p0, THETA, kc, vc, out, ws)
    else:
        sq.sq_kv_append(x, B, T, Hq, Hkv, p0, THETA, kc, vc)
        sq.sq_attention(x, B, T, Hq, Hkv, p0, THETA, kc, vc, out, ws)
    assert sq.sq_check() == 0
    got = out.float().cpu().numpy().astype(np.float64)
    for b in range(B):
        L = pos0[b] + T
        pos = np.arange(pos0[b], L)
        rows = qkv[b * T:(b + 1) * T].astype(np.float64)
        k = kc[b, :, :L].cpu().numpy().transpose(1, 0, 2).astype(np.float64)
        v = vc[b, :, :L].cpu().numpy().transpose(1, 0, 2).astype(np.float64)
        q = oracle.rope(rows[:, :Hq * D], pos, Hq, D, THETA).reshape(T, Hq, D)
        ref = oracle.attention(q, k, v, pos).reshape(T, Hq * D)
        assert_close(got[b * T:(b + 1) * T], ref, f"b={b}")


@pytest.mark.parametrize("T,Hq,Hkv", [(8, 1, 1), (9, 1, 1), (4, 8, 2), (17, 2, 2), (32, 2, 1), (13, 5, 1),
                                      (25, 8, 1), (1, 40, 8), (2, 5, 1)])
@pytest.mark.parametrize("ctx", [0, 63, 200])
@pytest.mark.parametrize("max_ctx", [256, 577])  # eight queries a CTA up to 512; an instance per query count
def test_query_counts(T, Hq, Hkv, ctx, max_ctx):
    _case(1, T, Hq, Hkv, [ctx], max_ctx, fused=T <= 9, seed=ctx)


@pytest.mark.parametrize("B,T,Hq,Hkv,max_ctx", [
    (2, 24, 16, 2, 512), (2, 25, 16, 2, 512),  # two CTAs of eight queries on an SM; one
    (1, 32, 6, 1, 64), (1, 32, 6, 1, 512),     # the most tokens: every group resident, and not
    (3, 7, 28, 4, 513), (3, 7, 28, 4, 512),    # the longest short cache, and one entry more
    (16, 7, 28, 4, 64), (24, 7, 28, 4, 64),    # two rounds of CTAs over one block; too many
])
@pytest.mark.parametrize("fused", [False, True])
def test_short_caches(B, T, Hq, Hkv, max_ctx, fused):
    _case(B, T, Hq, Hkv, [(37 * b) % (max_ctx - T + 1) for b in range(B - 1)] + [max_ctx - T], max_ctx, fused=fused,
          seed=T)


@pytest.mark.parametrize("ctx", [62, 63, 64, 127, 128])
def test_block_edges(ctx):
    _case(2, 2, 6, 2, [ctx, ctx + 1], 192, seed=ctx)
    _case(2, 2, 6, 2, [ctx, ctx + 1], 192, fused=True, seed=ctx)


@pytest.mark.parametrize("B,T,Hq,Hkv,pos0,max_ctx", [
    (1, 1, 5, 1, [19999], 20000),           # shares meet in the workspace
    (1, 20, 6, 2, [9001], 20000),           # ... two query groups, half the cache empty
    (2, 1, 12, 2, [4000, 3], 16384),        # the largest cluster
    (40, 1, 8, 8, [70 + i for i in range(40)], 128),  # one CTA per head
])
def test_shares_of_long_and_short_caches(B, T, Hq, Hkv, pos0, max_ctx):
    _case(B, T, Hq, Hkv, pos0, max_ctx, seed=B)


@pytest.mark.parametrize("qstd", [1e-4, 30.0])
def test_query_magnitudes(qstd):
    # the two fp16 terms of a query follow its own magnitude
    _case(1, 3, 4, 2, [100], 128, qstd=qstd)
