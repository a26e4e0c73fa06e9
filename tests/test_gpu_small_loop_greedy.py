"""Greedy targets of the one-launch generation loop: the LM head's tiles over CTAs and rounds, vocabularies that are no multiple of 16, equal logits.
Every emitted token is the oracle's choice up to the logit tolerance, and the statistics are those of a loop whose targets are these tokens."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs, inputs
from helpers import COUNTERS, LOGIT_TOL, counters_for_streams, greedy_margins, i32
from test_gpu_small_loop import CONFIGS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", ["0", "1"])
@pytest.mark.parametrize("head", ["plain", "copies", "larger copies"])
@pytest.mark.parametrize("name", list(CONFIGS))
def test_greedy_targets(name, head, small, monkeypatch):
    monkeypatch.setenv("CS_SMALL", small)
    cfg = CONFIGS[name]
    w = inputs.make_weights(cfg, seed=6, gain_jitter=0.05)
    half = cfg.vocab // 2
    if head != "plain":
        # the second half of the ids: logits equal to the first half's, which the lower id wins, or a quarter larger (the largest is about 1, the
        # tolerance 0.02), so that the winner is in the later tiles
        w["lm_head"][half:2 * half] = w["lm_head"][:half] * (1.0 if head == "copies" else 1.25)
    model = O.Model(cfg, w, contract=True)
    k, new, lens = 6, 24, [40, 23]
    ctx = cs.Context(cfg, inputs.weights_to(w, "cuda"), max_seq=80, max_batch=2, k_max=k)
    rng = np.random.default_rng(6)
    hists = [rng.integers(0, cfg.vocab, size=n) for n in lens]
    h = np.zeros((2, 72), np.int32)
    for b, row in enumerate(hists):
        h[b, :lens[b]] = row
    hd, n, kv, kvl = i32(h), i32(lens), ctx.alloc_kv(), torch.zeros(2, dtype=torch.int32, device="cuda")
    ctx.cs_prefill(hd, n, max(lens), kv, kvl)
    st = ctx.cs_decode_loop(hd, n, kv, kvl, 2, k, new)
    assert ctx.workspace_guards_intact()
    ctx.close()
    assert n.tolist() == [x + new for x in lens] and kvl.tolist() == [x + new - 1 for x in lens]
    gens = [hd[b, x:x + new].tolist() for b, x in enumerate(lens)]
    for row, gen in zip(hists, gens):
        assert max(greedy_margins(model, cfg, row, gen)) < LOGIT_TOL
        if head == "copies":
            assert not any(half <= t < 2 * half for t in gen)
        if head == "larger copies":
            assert half <= min(gen)
    want = counters_for_streams(hists, gens, 2, k)
    for key in COUNTERS:
        assert st[key] == want[key], key
    assert st["tau_hist"][:k + 1] == want["tau_hist"][:k + 1]
