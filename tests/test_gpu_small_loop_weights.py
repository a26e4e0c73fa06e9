"""Softmax weights below 2^-126 in the generation loop of a small model, in one launch and launch by launch: they are subnormal, not nothing.  The keys that get all of
the softmax have no values here, and those of a weight near 2^-127 have values near 2^123, so the attention output is made of such weights alone.

Tolerance: weights enter products as bf16 terms, whose last place is 2^-133 below 2^-126: half of one in 2^-127.5 is 1.1 % (at most, and alike for a row's
equal weights); a merge of shares weighs in fp32 and adds nothing to that.  Without them the rows are off by their whole size."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", ["0", "1"])
@pytest.mark.parametrize("every", [16, 64])          # a strong key in every block of keys that a warp takes / in the first one
def test_subnormal_weights_count(every, small, monkeypatch):
    monkeypatch.setenv("CS_SMALL", small)
    cfg, n, k, new, tok = inputs.TINY, 64, 3, 8, 5
    H, Dh = cfg.n_heads, cfg.head_dim
    w = inputs.make_weights(cfg, seed=4)
    model = O.Model(cfg, w, contract=True)
    # one token throughout: the queries of a head are the same up to their rotation, which hardly moves the dims of low frequency
    q = O.rmsnorm(model.embed([tok]), model._w(0, "attn_norm"), cfg.rms_eps) @ model._w(0, "wqkv")[:H * Dh].T
    q = O.rope(q.reshape(1, H, Dh), np.array([n + new // 2]), cfg.rope_theta)[0]
    slow = np.arange(Dh) % (Dh // 2) >= 12
    u = q * slow / (q * q * slow).sum(axis=1, keepdims=True)        # a key with a score of 1
    strong = np.arange(n) % every == 0
    score = np.where(strong, 64.0, 64.0 - 127.3) * np.log(2.0) * np.sqrt(Dh)
    cache = O.KVCache(cfg, 1, n + new + 1)
    rng = np.random.default_rng(0)
    cache.a[:, :, 0, :, :n] = O.round_bf16(rng.standard_normal((cfg.n_layers, 2, H, n, Dh)))
    cache.a[0, 0, 0, :, :n] = O.round_bf16(u[:, None, :] * score[None, :, None])
    cache.a[0, 1, 0, :, :n] *= np.where(strong, 0.0, 2.0 ** 123)[None, :, None]
    ctx = cs.Context(cfg, inputs.weights_to(w, "cuda"), max_seq=n + new + k + 1, max_batch=1, k_max=k)
    kv = ctx.alloc_kv()
    kv[:, :, 0, :, :n] = torch.from_numpy(cache.a[:, :, 0, :, :n].astype(np.float32)).to("cuda", torch.bfloat16)
    h, ln, kvl = i32(np.full((1, n + new + k + 1), tok)), i32([n + 1]), i32([n])
    ctx.cs_decode_loop(h, ln, kv, kvl, 3, k, new, script=i32(np.full((1, new), tok)))
    got = kv[1, :, 0, :, n:n + new].double().cpu().numpy()
    ctx.close()
    model.forward_block([tok] * new, n, cache, 0)
    want = cache.a[1, :, 0, :, n:n + new].astype(np.float64)
    assert np.linalg.norm(got - want) <= 0.015 * np.linalg.norm(want)
