"""Batches that leave one key slice per KV head: the tcgen05 attention kernels write the merged output themselves.  Against the mma.sync kernel with
its merge launch, on ragged lengths, ragged drafts, sequences without room (dead rows) and blocks at the edges of the kernels' row groups.

Tolerance: as between the kernels elsewhere - two-term operands, other orders of fp32 sums, K/V rows that round the other way (2^-8 of a
value, one of many keys) - no logit moves by more than 2^-8 of the largest."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu

CFG = inputs.ModelConfig(n_layers=2, d_model=256, n_heads=16, n_kv_heads=8, head_dim=128, d_ffn=512, vocab=640, rope_theta=500000.0, rms_eps=1e-5)


@pytest.mark.parametrize("B,k,keys", [(10, 0, 300), (10, 15, 1000), (16, 11, 700), (16, 15, 130), (18, 7, 2500), (12, 20, 257)])
def test_one_slice_agrees_with_merged_slices(B, k, keys, monkeypatch):
    w = inputs.weights_to(inputs.make_weights(CFG, seed=11, gain_jitter=0.05), "cuda")
    rng = np.random.default_rng(B + k)
    lens = [keys] + [int(x) for x in rng.integers(0, keys + 1, size=B - 1)]
    dlen = [int(x) for x in rng.integers(0, k + 1, size=B)]
    lens[2] = keys + 8                               # (with its draft beyond the cache's end)
    dlen[2] = k
    max_seq = keys + 8 + k
    last, draft = i32(rng.integers(0, CFG.vocab, size=B)), i32(rng.integers(0, CFG.vocab, size=(B, k)))
    kv0 = inputs.synthetic_kv(CFG, B, max_seq, max_seq, seed=3, device="cuda")
    outs = {}
    for kern in ("mma", "tc", "tcw"):
        monkeypatch.setenv("CS_ATTN_KERNEL", kern)
        ctx = cs.Context(CFG, w, max_seq=max_seq, max_batch=B, k_max=max(k, 1))
        kv, kvl = kv0.clone(), i32(lens)
        logits = torch.zeros(B, k + 1, CFG.vocab, dtype=torch.float32, device="cuda")
        ctx.cs_verify_step(last, draft, i32(dlen), kv, kvl, logits_dbg=logits)
        assert ctx.cs_sync_status() == cs.CS_ERR_CAPACITY and ctx.workspace_guards_intact()
        outs[kern] = ([logits[b, :dlen[b] + 1] for b in range(B) if b != 2], kv.float())
        ctx.close()
    for kern in ("tc", "tcw"):
        for a, c in zip(outs["mma"][0], outs[kern][0]):
            assert torch.isfinite(c).all() and float((a - c).abs().max()) <= float(a.abs().max()) / 256
        assert float((outs["mma"][1] - outs[kern][1]).abs().max()) <= float(outs["mma"][1].abs().max()) / 128
