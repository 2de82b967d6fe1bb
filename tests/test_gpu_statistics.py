"""GPU parity of the row statistics behind the accept step (bit exact against
the oracle): vocabularies at the edges of a CTA's, a cluster's and the
registers' share of a row, few and many rows (the two cluster sizes), rows off
the 16-byte grid, logits far apart; and a rejection whose residual has no mass."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_21704_gb300 as sq

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dev())


@pytest.mark.parametrize("R,V,std,T", [
    (1, 2048, 3.0, 1.0), (2, 2049, 3.0, 1.0), (40, 2047, 3.0, 1.0), (40, 16385, 20.0, 1.0),
    (3, 32769, 2.0, 0.05), (1, 327681, 3.0, 1.0), (39, 163841, 2.0, 1.0), (2, 1000001, 2.0, 1.5),
])
def test_softmax_edges_bit_exact(R, V, std, T):
    z = np.random.default_rng(R * V).normal(0, std, (R, V)).astype(np.float16)
    z[-1, -1] = np.float16(-60000.0)
    ws = torch.zeros(sq.sq_softmax_workspace_bytes(R, V), dtype=torch.uint8, device=dev())
    p = torch.empty(R, V, dtype=torch.float32, device=dev())
    sq.sq_softmax(_t(z), T, p, ws)
    assert sq.sq_check() == 0
    rows = range(R) if R <= 3 else [0, R // 2, R - 1]
    for r in rows:
        got = p[r].cpu().numpy()
        assert np.array_equal(got.view(np.uint32), oracle.softmax_row(z[r], T).view(np.uint32)), f"row {r}"


@pytest.mark.parametrize("B,V", [(1, 3000), (32, 40000)])
def test_rejection_without_residual_mass(B, V):
    # the draft's rows equal the parent's, and the draft token has probability
    # zero in both: rejected, with an empty residual, so p itself is drawn from
    rng = np.random.default_rng(B)
    zp = rng.normal(0, 2.0, (B, 3, V)).astype(np.float16)
    zp[:, :, 17] = np.float16(-60000.0)
    zq = np.ascontiguousarray(np.transpose(zp[:, :2], (1, 0, 2)))
    draft = np.full((B, 2), 17, np.int32)
    draft[: B // 2, 0] = np.argmax(zp[: B // 2, 0], axis=1)
    u = rng.random((B, 3)).astype(np.float32)
    ws = torch.zeros(sq.sq_accept_logits_workspace_bytes(B, 2, V), dtype=torch.uint8, device=dev())
    n = torch.empty(B, dtype=torch.int32, device=dev())
    tok = torch.empty(B, 3, dtype=torch.int32, device=dev())
    sq.sq_accept_logits(_t(zp), _t(zq), _t(draft), _t(u), 1.0, sq.SQ_ACCEPT_SAMPLE, n, tok, ws)
    assert sq.sq_check() == 0
    _, on, otok = oracle.accept_logits(zp, zq, draft, u, 1.0)
    assert set(on.tolist()) <= {0, 1}
    assert np.array_equal(n.cpu().numpy(), on) and np.array_equal(tok.cpu().numpy(), otok)
