"""The two-SM projections at the heights where their operands change form (32 | 33 rows: one-SM or
two-SM tiles; 128 | 129: stacked or separate bf16 terms; 256: the limit) and at widths whose tiles are
cut between SM pairs, against fp64 and the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import inputs
from helpers import LOGIT_TOL, argmax_consistent, i32, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 16, 33, 128, 129, 256])
def test_streamed_argmax_with_tiles_cut_between_pairs(rows):
    # 150 tiles of 256 ids over some 74 pairs, 9 K blocks each (the last one 8 wide): most runs start
    # inside a tile; the last tile holds 77 ids
    cfg = inputs.ModelConfig(n_layers=1, d_model=520, n_heads=4, n_kv_heads=4, head_dim=32, d_ffn=512, vocab=256 * 149 + 77)
    ctx, _ = make_pair(cfg, 64, 1, 10, seed=rows)
    g = torch.Generator().manual_seed(rows)
    X = torch.randn(rows, cfg.d_model, generator=g).to(torch.bfloat16)
    Xd = torch.zeros((rows + 15) // 16 * 16, cfg.d_model, dtype=torch.bfloat16, device="cuda")
    Xd[:rows] = X.cuda()
    logits = torch.zeros(rows, cfg.vocab, dtype=torch.float32, device="cuda")
    W = ctx.weights["lm_head"].cpu().double()
    want = (X.double() @ W.T).numpy()
    for _ in range(3):                       # the hand-over flags are back at rest after every launch
        ids = ctx.cs_lm_head(Xd, rows=rows, logits_dbg=logits)
        assert ctx.cs_sync_status() == 0
        # exact bf16 products, 520 fp32 additions: K * 2^-24 * sum |x w| bounds the error
        bound = cfg.d_model * 2.0 ** -24 * (X.double().abs() @ W.abs().T).numpy()
        assert (np.abs(logits.cpu().double().numpy() - want) <= bound).all()
        assert not argmax_consistent(want, ids.cpu().tolist(), tol=2 * float(bound.max()))
    assert ctx.workspace_guards_intact()
    ctx.close()


@pytest.mark.parametrize("B,k", [(2, 15), (3, 10), (8, 15), (3, 42), (16, 15)])   # 32, 33, 128, 129, 256 rows
def test_forward_at_every_operand_form(B, k):
    # d_ffn 9,608: 76 tiles of 128 gate/up pairs (the last one ragged), cut between the SM pairs
    cfg = inputs.ModelConfig(n_layers=1, d_model=264, n_heads=4, n_kv_heads=2, head_dim=128, d_ffn=9608, vocab=1000, rope_theta=500000.0)
    ctx, model = make_pair(cfg, 128, B, k, seed=1, gain_jitter=0.1)
    rng = np.random.default_rng(B)
    lens = [30 + b for b in range(B)]
    kv = inputs.synthetic_kv(cfg, B, 128, max(lens), seed=3, device="cuda")
    last, draft, dl, script = inputs.verify_inputs_with_tau(rng, B, k, rng.integers(0, k + 1, size=B), cfg.vocab)
    logits = torch.zeros(B, k + 1, cfg.vocab, dtype=torch.float32, device="cuda")
    cache = O.KVCache(cfg, B, 128)
    cache.a[...] = kv.float().cpu().numpy()
    al, ot, am = ctx.cs_verify_step(i32(last), i32(draft), i32(dl), kv, i32(lens), target_script=i32(script), logits_dbg=logits)
    assert ctx.cs_sync_status() == 0
    for b in range(B):
        tau, out, _, _, lg = O.verify_step(model, cache, b, last[b], draft[b], lens[b], script_row=script[b])
        assert int(al[b]) == tau and ot[b, :tau + 1].tolist() == out
        assert np.abs(logits[b].cpu().numpy() - lg).max() <= LOGIT_TOL
        assert not argmax_consistent(lg, am[b].tolist())
    assert ctx.workspace_guards_intact()
    ctx.close()
