"""Greedy targets of a small model whose LM head has rows that are NaN, in one launch and launch by launch: such an id is never the choice, and where no id
is left the target is -1."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs, inputs
from helpers import COUNTERS, LOGIT_TOL, counters_for_streams, greedy_margins, i32
from test_gpu_small_loop import CONFIGS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", ["0", "1"])
@pytest.mark.parametrize("nan", ["one id in five", "half of every tile", "all but one tile", "all"])
@pytest.mark.parametrize("name", ["tiny", "eight", "wide"])
def test_nan_is_nobodys_choice(name, nan, small, monkeypatch):
    monkeypatch.setenv("CS_SMALL", small)
    cfg = CONFIGS[name]
    ids = np.arange(cfg.vocab)
    # (ids of a tile of 16 are worked out in pairs, 8 apart)
    bad = {"one id in five": ids % 5 == 0, "half of every tile": ids % 16 < 8, "all but one tile": ids // 16 != 20, "all": ids >= 0}[nan]
    w = inputs.make_weights(cfg, seed=8, gain_jitter=0.05)
    known = dict(w)                      # the same choice without NaN: a row that must not be chosen repeats one that may
    if nan != "all":
        good = ids[~bad]
        known["lm_head"] = w["lm_head"].clone()
        known["lm_head"][bad] = w["lm_head"][torch.as_tensor(good[ids[bad] % len(good)])]
    w["lm_head"] = w["lm_head"].clone()
    w["lm_head"][bad] = float("nan")
    k, new, lens = 6, 20, [40, 23]
    ctx = cs.Context(cfg, inputs.weights_to(w, "cuda"), max_seq=80, max_batch=2, k_max=k)
    rng = np.random.default_rng(8)
    hists = [rng.integers(0, cfg.vocab, size=n) for n in lens]
    h = np.zeros((2, 72), np.int32)
    for b, row in enumerate(hists):
        h[b, :lens[b]] = row
    hd, n, kv, kvl = i32(h), i32(lens), ctx.alloc_kv(), torch.zeros(2, dtype=torch.int32, device="cuda")
    ctx.cs_prefill(hd, n, max(lens), kv, kvl)
    st = ctx.cs_decode_loop(hd, n, kv, kvl, 2, k, new)
    assert ctx.workspace_guards_intact()
    ctx.close()
    assert n.tolist() == [x + new for x in lens]
    gens = [hd[b, x:x + new].tolist() for b, x in enumerate(lens)]
    for row, gen in zip(hists, gens):
        if nan == "all":
            assert gen == [-1] * new
        else:
            assert not bad[gen].any() and min(gen) >= 0
            assert max(greedy_margins(O.Model(cfg, known, contract=True), cfg, row, gen)) < LOGIT_TOL
    want = counters_for_streams(hists, gens, 2, k)
    for key in COUNTERS:
        assert st[key] == want[key], key
