"""Rooms that no history has: more new tokens than an int adds up to are refused like any others that do not fit, and nothing is written."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", ["0", "1"])
@pytest.mark.parametrize("max_new", [(1 << 31) - 1, (1 << 31) - 60, (1 << 31) - 75, 1 << 30, 77])
def test_more_than_any_room(max_new, small, monkeypatch):
    monkeypatch.setenv("CS_SMALL", small)
    cfg = inputs.TINY
    ctx = cs.Context(cfg, inputs.weights_to(inputs.make_weights(cfg, seed=0), "cuda"), max_seq=200, max_batch=2, k_max=10)
    h = i32(np.random.default_rng(0).integers(0, cfg.vocab, size=(2, 136)))
    n, kv, kvl = i32([60, 61]), inputs.synthetic_kv(cfg, 2, 200, 60, seed=0, device="cuda"), i32([59, 60])
    before = [t.clone() for t in (h, n, kv, kvl)]
    with pytest.raises(cs.CsError) as e:
        ctx.cs_decode_loop(h, n, kv, kvl, 3, 10, max_new)
    assert e.value.code == cs.CS_ERR_CAPACITY and ctx.cs_sync_status() == cs.CS_OK
    assert all(torch.equal(a, b) for a, b in zip((h, n, kv, kvl), before)) and ctx.workspace_guards_intact()
    ctx.close()
