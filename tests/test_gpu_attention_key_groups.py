"""The mma.sync attention (head sizes 32 and 64) where its warps change between rows of their own and
shared rows with divided keys - 16 | 17 and 32 | 33 query rows per KV head, 64 | 65 rows for a second
CTA - with key ranges around its 64-key tiles, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import inputs
from helpers import LOGIT_TOL, i32, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim", [32, 64])
@pytest.mark.parametrize("rows,n", [(1, 2), (1, 64), (8, 65), (9, 63), (16, 129), (17, 128), (32, 200), (33, 190)])
def test_rows_and_keys_at_the_edges(head_dim, rows, n):
    cfg = inputs.ModelConfig(n_layers=2, d_model=128, n_heads=4, n_kv_heads=2, head_dim=head_dim, d_ffn=256,
                             vocab=500, rope_theta=10000.0, rms_eps=1e-5)
    B, k = 2, rows - 1
    lens = [n, max(1, n // 2)]
    max_seq = n + rows + 5
    ctx, model = make_pair(cfg, max_seq, B, max(k, 1), seed=rows, gain_jitter=0.1)
    rng = np.random.default_rng(n)
    hist = rng.integers(0, cfg.vocab, size=(B, n + 3), dtype=np.int32)
    draft = rng.integers(0, cfg.vocab, size=(B, k), dtype=np.int32)
    kv = ctx.alloc_kv()
    kv_len = torch.zeros(B, dtype=torch.int32, device="cuda")
    ctx.cs_prefill(i32(hist), i32(lens), n, kv, kv_len)
    last = [int(hist[b, lens[b] - 1]) for b in range(B)]
    dr = i32(draft) if k > 0 else torch.zeros((B, 0), dtype=torch.int32, device="cuda")
    logits = torch.zeros(B, rows, cfg.vocab, dtype=torch.float32, device="cuda")
    ctx.cs_verify_step(i32(last), dr, i32([k] * B), kv, kv_len, logits_dbg=logits)
    assert ctx.cs_sync_status() == 0
    for b in range(B):
        cache = O.KVCache(cfg, 1, max_seq)
        seq = hist[b, :lens[b]].tolist() + draft[b].tolist()
        want = model.forward_block(seq, 0, cache, 0)[lens[b] - 1:]
        assert float(np.abs(logits[b].cpu().numpy() - want).max()) < LOGIT_TOL
    ctx.close()
