"""The generation loop of a small model in one launch, at the sizes where it can go wrong: rows at the edges of its quarters of four tokens, clusters
of eight and sixteen, tiles dealt out unevenly, several tiles a warp, K longer than a warp's ring, grouped heads, blocks of keys at their edges,
vocabularies that are no multiple of 16, searches with every key length, sequences that stop at different steps.  Against a launch per kernel
(CS_SMALL=0) on the same inputs: tokens, lengths and statistics are the same, cached rows agree.

Tolerance of the cached rows: both carry activations as two bf16 terms and sum in fp32, in another order, so the first layer agrees to about 2^-15;
what this moves across a rounding boundary of bf16 differs by one step, 2^-7 of the largest value at most."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu


def _cfg(layers, d, heads, kv_heads, dh, ffn, vocab):
    return inputs.ModelConfig(n_layers=layers, d_model=d, n_heads=heads, n_kv_heads=kv_heads, head_dim=dh, d_ffn=ffn, vocab=vocab)


CONFIGS = {
    "tiny": inputs.TINY,
    "eight": _cfg(3, 160, 4, 2, 32, 288, 1003),      # clusters of eight, ten tiles and nine blocks of SwiGLU over eight CTAs
    "idle": _cfg(2, 288, 6, 3, 32, 544, 2000),       # four CTAs without a KV head; K blocks of 64 that are half full
    "gqa64": _cfg(1, 256, 4, 2, 64, 512, 777),
    "wide": _cfg(2, 544, 4, 4, 64, 512, 5000),       # K longer than a ring, three tiles a CTA, LM-head tiles in several rounds
    "mqa": _cfg(1, 256, 4, 1, 32, 512, 1500),        # sixteen CTAs share a KV head
}


def _loop(cfg, w, small, hists, scripts, lens, k, max_new, max_seq, stride, gamma, policy, monkeypatch):
    monkeypatch.setenv("CS_SMALL", small)
    B = len(hists)
    ctx = cs.Context(cfg, w, max_seq=max_seq, max_batch=B, k_max=k)
    h, s = np.zeros((B, stride), np.int32), np.zeros((B, max_new), np.int32)
    for b in range(B):
        h[b, :len(hists[b])], s[b] = hists[b], scripts[b][:max_new]
    kv = inputs.synthetic_kv(cfg, B, max_seq, max(lens), seed=3, device="cuda")
    kv[:, :, :, :, max(lens):] = float("nan")        # (rows that nobody has written must not be read)
    # in a batch of three and more the last cache does not go with its history: refused, while the others run
    hd, n, kvl = i32(h), i32([x + 1 for x in lens]), i32(lens if B < 3 else lens[:-1] + [lens[-1] - 1])
    status = cs.CS_OK
    try:
        st = ctx.cs_decode_loop(hd, n, kv, kvl, gamma, k, max_new, policy=policy, script=i32(s))
    except cs.CsError as e:
        status, st = e.code, None
    assert ctx.workspace_guards_intact()
    ctx.close()
    return hd, n, kvl, st, kv, status


@pytest.mark.parametrize("B,k,n,gamma,policy", [(1, 0, 31, 1, cs.LATEST), (1, 3, 48, 3, cs.LATEST), (3, 4, 200, 2, cs.FIRST), (2, 8, 1023, 3, cs.LATEST),
                                                (9, 11, 130, 5, cs.LATEST), (1, 12, 64, 8, cs.FIRST), (2, 15, 257, 3, cs.LATEST)])
@pytest.mark.parametrize("name", list(CONFIGS))
def test_agrees_with_a_launch_per_kernel(name, B, k, n, gamma, policy, monkeypatch):
    cfg = CONFIGS[name]
    w = inputs.weights_to(inputs.make_weights(cfg, seed=4, gain_jitter=0.05), "cuda")
    rng = np.random.default_rng(n + k)
    lens = [n - 5 * b for b in range(B)]
    # a small alphabet: matches, partial acceptance and drafts clipped at the history's end
    hists = [rng.integers(0, 3, size=m + 1) for m in lens]
    max_new = 3 * k + 4
    scripts = [rng.integers(0, 3, size=max_new) for _ in range(B)]
    args = (hists, scripts, lens, k, max_new, n + 1 + max_new + k, n + 1 + max_new + (k & 1), gamma, policy, monkeypatch)
    want, got = _loop(cfg, w, "0", *args), _loop(cfg, w, "1", *args)
    for a, b in zip(want[:3], got[:3]):
        assert torch.equal(a, b)
    assert want[3] == got[3] and want[5] == got[5] == (cs.CS_ERR_ARG if B >= 3 else cs.CS_OK)
    assert torch.equal(want[4].isnan(), got[4].isnan())
    a, b = want[4].float().nan_to_num(), got[4].float().nan_to_num()
    assert float((a - b).abs().max()) <= float(a.abs().max()) / 128


def test_is_taken_by_default_on_small_models_only(monkeypatch):
    """What tells the two forms apart from outside is the order of their sums: the cached rows differ somewhere."""
    cfg = CONFIGS["tiny"]
    w = inputs.weights_to(inputs.make_weights(cfg, seed=4), "cuda")
    rng = np.random.default_rng(0)
    args = ([rng.integers(0, 50, size=201)], [rng.integers(0, 50, size=30)], [200], 10, 30, 260, 260, 3, cs.LATEST, monkeypatch)
    rows = {small: _loop(cfg, w, small, *args)[4].float().nan_to_num() for small in ("0", "1", "")}
    assert torch.equal(rows["1"], rows[""]) and not torch.equal(rows["0"], rows["1"])


@pytest.mark.parametrize("unit", range(7))
def test_a_hand_over_that_never_comes(unit, monkeypatch):
    """Every wait for another CTA runs out after the context's limit: the call reports it, and the context goes on."""
    monkeypatch.setenv("CS_WAIT_LIMIT_US", "2000")
    cfg = CONFIGS["tiny"]
    w = inputs.weights_to(inputs.make_weights(cfg, seed=4), "cuda")
    ctx = cs.Context(cfg, w, max_seq=300, max_batch=2, k_max=4)
    rng = np.random.default_rng(1)
    h, script = i32(rng.integers(0, 50, size=(2, 300))), i32(rng.integers(0, 50, size=(2, 20)))
    kv = inputs.synthetic_kv(cfg, 2, 300, 200, seed=3, device="cuda")
    n = i32([201, 190])
    ctx.cs_debug_drop_chain_tile(unit)
    with pytest.raises(cs.CsError) as e:
        ctx.cs_decode_loop(h, n, kv, n - 1, 3, 4, 20, script=script)
    assert e.value.code == cs.CS_ERR_TIMEOUT and ctx.cs_sync_status() == cs.CS_OK
    n = i32([201, 190])
    st = ctx.cs_decode_loop(h, n, kv, n - 1, 3, 4, 20, script=script)
    assert st["emitted"] == 40 and torch.equal(h[0, 201:221], script[0]) and torch.equal(h[1, 190:210], script[1])
    assert ctx.workspace_guards_intact()
    ctx.close()
