"""Bounded waits of the two-SM projections that run out.  The limit is 2 ms for these contexts and a
launch leaves out one K block: the MMA warp of a pair waits for a tile that never arrives, the odd
CTA for an accumulator, and in the streamed form a pair that is whole for sums of one that gave up.
Nothing faults or hangs; the host reads CS_ERR_TIMEOUT and the next call is right: the words by which
pairs hand sums over are back at rest."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import make_pair

pytestmark = pytest.mark.gpu

# 150 tiles of 256 ids over some 74 pairs, 9 K blocks each: most runs start and end inside a tile
CFG = inputs.ModelConfig(n_layers=1, d_model=520, n_heads=4, n_kv_heads=4, head_dim=32, d_ffn=512, vocab=256 * 149 + 77)


def _timed(call):
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record()
    out = call()
    ev1.record()
    torch.cuda.synchronize()
    return out, ev0.elapsed_time(ev1)


@pytest.mark.parametrize("rows", [1, 40, 256])          # read out in one step, by four groups, two operands per term
@pytest.mark.parametrize("k_block", [0, 7, 15])         # in a handed-over tail, later, behind the ring's first turn
def test_streamed_projection(monkeypatch, rows, k_block):
    monkeypatch.setenv("CS_WAIT_LIMIT_US", "2000")
    ctx, _ = make_pair(CFG, 64, 1, 10)
    X = torch.randn((rows + 15) // 16 * 16, CFG.d_model, device="cuda").to(torch.bfloat16)

    def head(dst):
        return ctx.cs_lm_head(X, rows=rows, logits_dbg=dst)

    want = torch.zeros(rows, CFG.vocab, dtype=torch.float32, device="cuda")
    want_ids = head(want)
    assert ctx.cs_sync_status() == cs.CS_OK
    for _ in range(2):
        got = torch.full_like(want, float("nan"))
        ctx.cs_debug_drop_tile(k_block)
        _, ms = _timed(lambda: head(got))
        assert 1.0 <= ms <= 500.0                        # about the limit, not 2 s, and returned
        assert ctx.cs_sync_status() == cs.CS_ERR_TIMEOUT
        # what is there is right: a pair that gave up writes nothing, never part of a sum
        there = ~torch.isnan(got)
        assert bool(there.any()) and not bool(there.all()) and torch.equal(got[there], want[there])
        assert ctx.cs_sync_status() == cs.CS_OK          # reported once
        got = torch.zeros_like(want)
        assert torch.equal(head(got), want_ids) and torch.equal(got, want)
        assert ctx.cs_sync_status() == cs.CS_OK
    assert ctx.workspace_guards_intact()
    ctx.close()


@pytest.mark.parametrize("rows", [33, 200])
@pytest.mark.parametrize("K", [256, 4096])               # one pair per tile; several that share its K blocks
def test_split_projection(monkeypatch, rows, K):
    monkeypatch.setenv("CS_WAIT_LIMIT_US", "2000")
    ctx, _ = make_pair(CFG, 64, 1, 10)
    X = torch.randn((rows + 15) // 16 * 16, K, device="cuda").to(torch.bfloat16)
    W = torch.randn(300, K, device="cuda").to(torch.bfloat16)
    want = ctx.cs_linear(X, W, rows=rows)
    assert ctx.cs_sync_status() == cs.CS_OK
    for _ in range(2):
        ctx.cs_debug_drop_tile(2)
        got, ms = _timed(lambda: ctx.cs_linear(X, W, rows=rows))
        assert 1.0 <= ms <= 500.0 and ctx.cs_sync_status() == cs.CS_ERR_TIMEOUT
        if K == 256:
            assert float(got.abs().max()) == 0.0         # zeros, never partial sums
        assert torch.equal(ctx.cs_linear(X, W, rows=rows), want) and ctx.cs_sync_status() == cs.CS_OK
    assert ctx.workspace_guards_intact()
    ctx.close()


def test_forward_after_a_timeout_nobody_asked_about(monkeypatch):
    """Clients that never take a status: the forward after the one that timed out is right."""
    monkeypatch.setenv("CS_WAIT_LIMIT_US", "2000")
    ctx, _ = make_pair(CFG, 96, 2, 4)
    kv0 = inputs.synthetic_kv(CFG, 2, 96, 40, seed=3, device="cuda")
    rng = np.random.default_rng(4)
    hist = torch.from_numpy(rng.integers(0, CFG.vocab, size=(2, 40)).astype(np.int32)).cuda()
    len40 = torch.full((2,), 40, dtype=torch.int32, device="cuda")

    def step():
        kv, logits = kv0.clone(), torch.zeros(2, 5, CFG.vocab, dtype=torch.float32, device="cuda")
        out = ctx.cs_verify_step(hist[:, 0].contiguous(), hist[:, 1:5].contiguous(), torch.full_like(len40, 4), kv, len40.clone(), logits_dbg=logits)
        return [kv, logits, *out]

    def prefill():
        kv = torch.zeros_like(kv0)
        ctx.cs_prefill(hist, len40, 40, kv, torch.zeros_like(len40))
        return [kv]

    X = torch.randn(256, CFG.d_model, device="cuda").to(torch.bfloat16)
    want = step(), prefill()
    assert ctx.cs_sync_status() == cs.CS_OK
    words = ctx._raw[ctx._ws_off:ctx._ws_off + ctx.workspace_bytes].view(torch.int32)
    for call, expect in zip((step, prefill), want):
        for rows in (16, 256):
            ctx.cs_lm_head(X, rows=rows)
            rest = words.clone()
            ctx.cs_debug_drop_tile(0)
            ctx.cs_lm_head(X, rows=rows)                 # every second pair gives up and does not take its neighbours' sums
            raised = (rest == 0) & (words == 1)          # (few other words of the workspace go from 0 to 1 here)
            assert int(raised.sum()) >= 20
            got = call()
            assert not bool(words[raised].any())
            assert ctx.cs_sync_status() == cs.CS_ERR_TIMEOUT
            assert all(torch.equal(a, b) for a, b in zip(got, expect))
    ctx.close()
