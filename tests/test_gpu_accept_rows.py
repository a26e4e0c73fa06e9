"""Acceptance at the block sizes where its division of warps changes (one row on all 32 warps, 8 | 9,
16 | 17 and 32 | 33 rows, 256 rows): greedy tokens, accepted length and emitted tokens are whole
numbers and must be exactly what the logits and the draft say."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu

CFG = inputs.TINY


@pytest.mark.parametrize("B,k", [(1, 0), (1, 7), (1, 8), (3, 15), (2, 16), (1, 31), (1, 32), (1, 255), (16, 15)])
def test_acceptance_follows_the_logits(B, k):
    rng = np.random.default_rng(k)
    w = inputs.weights_to(inputs.make_weights(CFG, seed=3), "cuda")
    n = 50
    ctx = cs.Context(CFG, w, max_seq=n + k + 8, max_batch=B, k_max=max(k, 1))
    kv = inputs.synthetic_kv(CFG, B, n + k + 8, n, seed=4, device="cuda")
    last = rng.integers(0, CFG.vocab, size=B)
    draft = rng.integers(0, CFG.vocab, size=(B, k)).astype(np.int32)
    dl = np.array([max(0, k - 3 * b) for b in range(B)], dtype=np.int32)
    taus = set()
    for _ in range(4):                                 # every pass takes over what the last one predicted: prefixes grow
        logits = torch.zeros(B, k + 1, CFG.vocab, dtype=torch.float32, device="cuda")
        dr = i32(draft) if k > 0 else torch.zeros((B, 0), dtype=torch.int32, device="cuda")
        kvl = i32([n] * B)
        al, ot, am = (t.cpu().numpy() for t in ctx.cs_verify_step(i32(last), dr, i32(dl), kv, kvl, logits_dbg=logits))
        assert ctx.cs_sync_status() == 0
        want = logits.cpu().numpy().argmax(-1)
        for b in range(B):
            d = int(dl[b])
            assert am[b].tolist() == want[b, :d + 1].tolist() + [-1] * (k - d)
            tau = 0
            while tau < d and draft[b, tau] == want[b, tau]:
                tau += 1
            assert al[b] == tau and kvl[b].item() == n + tau + 1
            assert ot[b].tolist() == want[b, :tau + 1].tolist() + [-1] * (k - tau)
            taus.add(tau)
        draft = np.where(am[:, :k] >= 0, am[:, :k], draft).astype(np.int32)
    assert k == 0 or max(taus) >= min(3, int(dl.max()))
    ctx.close()
