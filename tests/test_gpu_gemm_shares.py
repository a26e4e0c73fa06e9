"""Tall projections whose K ranges are split between SM pairs: a pair that comes before all of its tile
have started leaves its share of the tokens to one that waits.  Which pairs do depends on when the
device starts them, so here it is set from the host: share 0, one in the middle, all but the last.
The sums keep their order whoever finishes a share, so everything is the same bit for bit."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import inputs
from helpers import i32, make_pair

pytestmark = pytest.mark.gpu

CFG = inputs.ModelConfig(n_layers=2, d_model=520, n_heads=16, n_kv_heads=4, head_dim=128, d_ffn=9608, vocab=1000, rope_theta=500000.0)


@pytest.mark.parametrize("B,k", [(3, 10), (3, 42), (16, 15)])   # 33, 129, 256 rows: one residual row ahead per thread, and several
def test_shares_left_to_other_pairs(B, k):
    ctx, _ = make_pair(CFG, 96, B, k, seed=5, gain_jitter=0.1)
    rng = np.random.default_rng(B)
    kv0 = inputs.synthetic_kv(CFG, B, 96, 40, seed=3, device="cuda")
    last, draft, dl, script = inputs.verify_inputs_with_tau(rng, B, k, rng.integers(0, k + 1, size=B), CFG.vocab)
    X = torch.randn(256, 2048, device="cuda").to(torch.bfloat16)
    W = torch.randn(130, 2048, device="cuda").to(torch.bfloat16)

    def run():
        kv, logits = kv0.clone(), torch.zeros(B, k + 1, CFG.vocab, dtype=torch.float32, device="cuda")
        out = ctx.cs_verify_step(i32(last), i32(draft), i32(dl), kv, i32([30 + b for b in range(B)]), target_script=i32(script), logits_dbg=logits)
        Y = ctx.cs_linear(X, W, rows=B * (k + 1))
        assert ctx.cs_sync_status() == 0
        return [kv, logits, Y, *out]

    want = run()
    for mask in (0b1, 0b10, 0b11, 0b1011, 0b1111111, 0):
        ctx.cs_debug_leave_shares(mask)
        for _ in range(2):               # (a second time: the words of the first are back at rest)
            for a, b in zip(run(), want):
                assert torch.equal(a, b), f"mask {mask:b}"
    assert ctx.workspace_guards_intact()
    ctx.close()
