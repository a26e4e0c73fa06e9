"""cs_decode_loop on a model large enough for it to capture its step while the first two run: tokens,
lengths, cache and statistics (whole numbers and bytes) must be those of the loop that enqueues every
step, for loops that end before, at and after the switch, for fresh buffers on every call, and in real
mode with an end-of-sequence token."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu

CFG = inputs.ModelConfig(n_layers=2, d_model=2048, n_heads=16, n_kv_heads=4, head_dim=128, d_ffn=4096, vocab=2000,
                         rope_theta=500000.0, rms_eps=1e-5)


def test_captured_steps_are_the_enqueued_ones(monkeypatch):
    w = inputs.weights_to(inputs.make_weights(CFG, seed=6), "cuda")
    B, n0, k = 2, 150, 5
    rng = np.random.default_rng(3)
    ctxt = rng.integers(0, 60, size=(B, n0)).astype(np.int32)
    calls = [(1, -1), (6, -1), (20, -1), (60, -1), (60, 7), (61, -1)]
    results = {}
    for ng in ("1", "0"):
        monkeypatch.setenv("CS_NO_GRAPH", ng)
        ctx = cs.Context(CFG, w, max_seq=n0 + 80, max_batch=B, k_max=k)
        out = []
        for max_new, eos in calls:
            h = np.zeros((B, n0 + 80), dtype=np.int32)
            h[:, :n0] = ctxt
            hist, hl = i32(h), i32([n0, n0 - 20])
            kv, kvl = ctx.alloc_kv(), torch.zeros(B, dtype=torch.int32, device="cuda")
            kv.zero_()
            ctx.cs_prefill(hist, hl, n0, kv, kvl)
            st = ctx.cs_decode_loop(hist, hl, kv, kvl, 3, k, max_new, eos_id=eos)
            assert ctx.cs_sync_status() == 0
            out.append((hist.cpu().tolist(), hl.cpu().tolist(), kvl.cpu().tolist(), {a: np.asarray(b).tolist() for a, b in st.items()}))
            if eos < 0:
                assert hl.cpu().tolist() == [n0 + max_new, n0 - 20 + max_new]
        results[ng] = out
        ctx.close()
    assert results["0"] == results["1"]
