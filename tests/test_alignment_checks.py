"""Pointers whose alignment the kernels rely on and that no operand map checks: refused on the host, before
anything is launched."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs


@pytest.mark.parametrize("name", ["embed", "final_norm", "attn_norm", "ffn_norm"])
def test_create_refuses_rows_off_their_boundary(name):
    lib, cfg = cs.load(), inputs.TINY
    c = cs.CsModelConfig(cfg.n_layers, cfg.d_model, cfg.n_heads, cfg.n_kv_heads, cfg.head_dim, cfg.d_ffn, cfg.vocab, 64, 1, 4, cfg.rope_theta, cfg.rms_eps)
    ok, off = 1 << 20, (1 << 20) + 4                     # (numbers: nothing is read before the checks)
    cw, keep = cs.CsWeights(), []
    for f in ("embed", "lm_head", "final_norm"):
        setattr(cw, f, off if f == name else ok)
    for f in ("attn_norm", "wqkv", "wo", "ffn_norm", "w_gate_up", "w_down"):
        keep.append((C.c_void_p * cfg.n_layers)(*[off if f == name and l == cfg.n_layers - 1 else ok for l in range(cfg.n_layers)]))
        setattr(cw, f, C.cast(keep[-1], C.POINTER(C.c_void_p)))
    h = C.c_void_p()
    assert lib.cs_create(C.byref(h), C.byref(c), C.byref(cw), C.c_void_p(1 << 20), lib.cs_workspace_bytes(C.byref(c))) == cs.CS_ERR_ARG
    assert b"aligned" in lib.cs_last_error(None)


@pytest.mark.gpu
@pytest.mark.parametrize("head_dim", [32, 128])
def test_calls_refuse_a_cache_off_its_boundary(head_dim):
    cfg = inputs.ModelConfig(n_layers=1, d_model=256, n_heads=2, n_kv_heads=2, head_dim=head_dim, d_ffn=512, vocab=512)
    w = inputs.weights_to(inputs.make_weights(cfg, seed=1), "cuda")
    ctx, draft = (cs.Context(cfg, w, max_seq=64, max_batch=1, k_max=4) for _ in range(2))
    good = ctx.alloc_kv()
    bad = torch.zeros(good.numel() + 8, dtype=torch.bfloat16, device="cuda")[4:4 + good.numel()].view(good.shape)   # 8 bytes off
    i32 = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")
    hist, hl, kl = i32([list(range(20)) + [0] * 20]), i32([20]), i32([19])
    host, hlen = hist.cpu(), hl.cpu()
    calls = [lambda kv: ctx.cs_prefill(hist, hl, 20, kv, kl),
             lambda kv: ctx.cs_verify_step(i32([3]), i32([[1, 2]]), i32([2]), kv, kl),
             lambda kv: ctx.cs_decode_loop(hist, hl, kv, kl, 3, 2, 4),
             lambda kv: ctx.cs_loop_begin(hist, hl, kv, kl, 3, 2, 4),
             lambda kv: ctx.cs_step_host(host, hlen, hist.clone(), hl.clone(), kv, kl, 3, 2, torch.zeros(1, dtype=torch.int32), torch.zeros(1, 3, dtype=torch.int32)),
             lambda kv: ctx.cs_decode_loop_drafted(draft, hist, hl, kv, kl, good, kl.clone(), 3, 2, 2, 4),
             lambda kv: ctx.cs_decode_loop_drafted(draft, hist, hl, good, kl, kv, kl.clone(), 3, 2, 2, 4)]
    for call in calls:
        with pytest.raises(cs.CsError) as err:
            call(bad)
        assert err.value.code == cs.CS_ERR_ARG and "aligned" in str(err.value)
    assert ctx.cs_sync_status() == cs.CS_OK and not bool(bad.any()) and int(hl[0]) == 20 and int(kl[0]) == 19
    ctx.close(); draft.close()
