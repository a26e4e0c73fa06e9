"""The chained projections of short blocks (one launch for everything between two attentions) at the sizes where
they can go wrong: rows at the edges of their three paddings, widths that are no multiple of the 128-feature tiles or
of the 64-wide K blocks, every head size, tiles shared by many runs and runs that hold several tiles.  Against a
launch per projection (CS_CHAIN=0) on the same inputs.

Tolerance: both carry activations as two bf16 terms and sum in fp32, in another order, so the first layer agrees to
about 2^-15; a K or V element of the next layers that this moves across a rounding boundary of bf16 differs by 2^-8 of
itself and is one of many keys, so no logit can move by more than 2^-8 of the largest, no cached value by more
than one bf16 step of the largest."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs, inputs
from helpers import LOGIT_TOL, i32, make_pair

pytestmark = pytest.mark.gpu


def _cfg(d, heads, kv_heads, dh, ffn, layers=3):
    return inputs.ModelConfig(n_layers=layers, d_model=d, n_heads=heads, n_kv_heads=kv_heads, head_dim=dh, d_ffn=ffn, vocab=777)


CONFIGS = {
    "ragged": _cfg(520, 5, 5, 32, 328),             # 4.06 tiles, 8.1 K blocks, a head group of 32 features at the end
    "tiny": _cfg(256, 8, 8, 32, 1024, layers=2),    # fewer runs than SMs
    "shared": _cfg(256, 16, 2, 128, 9000),          # tiles of down shared by 35 runs
    "wide": _cfg(2048, 16, 4, 64, 2048),            # gate/up: runs inside a tile; many key slices to merge
    "long": _cfg(256, 2, 1, 128, 20000),            # runs that hold several whole tiles
    "deep": _cfg(4104, 2, 1, 128, 328),             # norms of 33 tiles: their words, and the projections', beyond one window of 32
}
# at 32 rows the merge has more slices than a warp's first pass takes: 29 for one warp an item, 49 for two (keys)
SLICES = {"one warp": (_cfg(256, 20, 5, 128, 1024, layers=2), 4000), "two warps": (_cfg(256, 12, 3, 128, 1024, layers=2), 6500)}


def _step(cfg, w, B, k, kv_len, max_seq, alone, monkeypatch):
    monkeypatch.setenv("CS_CHAIN", "0" if alone else "1")
    ctx = cs.Context(cfg, w, max_seq=max_seq, max_batch=B, k_max=max(k, 1))
    rng = np.random.default_rng(k + kv_len)
    last, draft = i32(rng.integers(0, cfg.vocab, size=B)), i32(rng.integers(0, cfg.vocab, size=(B, k)))
    dlen = i32([max(0, k - 2 * b) for b in range(B)])
    kv = inputs.synthetic_kv(cfg, B, max_seq, kv_len, seed=3, device="cuda")
    lens = i32([kv_len - 5 * b for b in range(B)])
    outs = []
    for _ in range(2):                              # (the second forward finds the counters of the first)
        l, logits = lens.clone(), torch.zeros(B, k + 1, cfg.vocab, dtype=torch.float32, device="cuda")
        ctx.cs_verify_step(last, draft, dlen, kv, l, logits_dbg=logits)
        assert ctx.cs_sync_status() == cs.CS_OK
        outs.append(logits)
    assert torch.equal(outs[0], outs[1]) and ctx.workspace_guards_intact()
    ctx.close()
    return outs[0], kv.float(), [int(n) for n in dlen]


@pytest.mark.parametrize("B,k", [(1, 0), (1, 7), (1, 8), (2, 7), (1, 16), (4, 7)])
@pytest.mark.parametrize("name", list(CONFIGS))
def test_agrees_with_a_launch_per_projection(name, B, k, monkeypatch):
    cfg = CONFIGS[name]
    w = inputs.weights_to(inputs.make_weights(cfg, seed=4, gain_jitter=0.05), "cuda")
    kv_len = 900 if name == "wide" else 150
    want, kv_want, dlen = _step(cfg, w, B, k, kv_len, kv_len + 40, True, monkeypatch)
    got, kv_got, _ = _step(cfg, w, B, k, kv_len, kv_len + 40, False, monkeypatch)
    for b in range(B):                              # rows behind the draft attend to nothing
        a, c = want[b, :dlen[b] + 1], got[b, :dlen[b] + 1]
        assert float((a - c).abs().max()) <= float(a.abs().max()) / 256
    assert float((kv_want - kv_got).abs().max()) <= float(kv_want.abs().max()) / 128


@pytest.mark.parametrize("name", list(SLICES))
def test_merge_takes_its_slices_in_several_passes(name, monkeypatch):
    cfg, kv_len = SLICES[name]
    w = inputs.weights_to(inputs.make_weights(cfg, seed=4, gain_jitter=0.05), "cuda")
    want, kv_want, _ = _step(cfg, w, 1, 31, kv_len, kv_len + 40, True, monkeypatch)
    got, kv_got, _ = _step(cfg, w, 1, 31, kv_len, kv_len + 40, False, monkeypatch)
    assert float((want - got).abs().max()) <= float(want.abs().max()) / 256
    assert float((kv_want - kv_got).abs().max()) <= float(kv_want.abs().max()) / 128


@pytest.mark.parametrize("rows", [1, 11, 32])
@pytest.mark.parametrize("name", ["ragged", "shared", "long", "deep"])
def test_agrees_with_the_oracle(name, rows, monkeypatch):
    """Logits and appended keys and values against the 64-bit oracle; tolerances as for a launch per projection."""
    monkeypatch.setenv("CS_CHAIN", "1")
    cfg = inputs.ModelConfig(**{**CONFIGS[name].__dict__, "n_layers": 2})
    ctx, model = make_pair(cfg, 200, 1, 31, gain_jitter=0.05)
    kv_len = 70
    kv = inputs.synthetic_kv(cfg, 1, 200, kv_len, seed=3, device="cuda")
    cache = O.KVCache(cfg, 1, 200)
    cache.a[:, :, :, :, :kv_len] = kv[:, :, :, :, :kv_len].float().cpu().numpy()
    tok = np.random.default_rng(rows).integers(0, cfg.vocab, size=rows).astype(np.int32)
    logits = torch.zeros(1, rows, cfg.vocab, dtype=torch.float32, device="cuda")
    ctx.cs_verify_step(i32(tok[:1]), i32(tok[None, 1:]), i32([rows - 1]), kv, i32([kv_len]), logits_dbg=logits)
    assert ctx.cs_sync_status() == cs.CS_OK
    want = model.forward_block(tok.tolist(), kv_len, cache, 0)
    assert float(np.abs(logits[0].cpu().numpy() - want).max()) <= LOGIT_TOL
    new = slice(kv_len, kv_len + rows)
    assert float(np.abs(kv[:, :, 0, :, new].float().cpu().numpy() - cache.a[:, :, 0, :, new]).max()) <= 2e-2
    ctx.close()


@pytest.mark.parametrize("B,rows", [(1, 1), (1, 17), (1, 32), (3, 10), (2, 1)])
@pytest.mark.parametrize("name", ["ragged", "wide"])
def test_prefill_ends_in_a_short_chunk(name, B, rows, monkeypatch):
    """A chunk of full height (on SM pairs), then one that is chained: its last layer has neither a QKV projection nor
    a norm behind it.  A verify step over the cache follows."""
    cfg = CONFIGS[name]
    w = inputs.weights_to(inputs.make_weights(cfg, seed=4, gain_jitter=0.05), "cuda")
    n = 256 // B + rows + 1
    rng = np.random.default_rng(rows)
    hist, last, draft = rng.integers(0, cfg.vocab, size=(B, n + 7)), rng.integers(0, cfg.vocab, size=B), rng.integers(0, cfg.vocab, size=(B, 4))
    outs = []
    for switch in "01":
        monkeypatch.setenv("CS_CHAIN", switch)
        ctx = cs.Context(cfg, w, max_seq=n + 40, max_batch=B, k_max=4)
        kv, kvl, lens = ctx.alloc_kv(), i32(np.zeros(B)), i32([n] + [n - 1] * (B - 1))
        for _ in range(2):
            kv.zero_()
            ctx.cs_prefill(i32(hist), lens, n, kv, kvl)
        assert kvl.cpu().tolist() == [n - 1] + [n - 2] * (B - 1)
        logits = torch.zeros(B, 5, cfg.vocab, dtype=torch.float32, device="cuda")
        ctx.cs_verify_step(i32(last), i32(draft), i32([4] * B), kv, kvl, logits_dbg=logits)
        assert ctx.cs_sync_status() == cs.CS_OK and ctx.workspace_guards_intact()
        outs.append((logits, kv.float()))
        ctx.close()
    for a, c, share in zip(outs[0], outs[1], (256, 128)):
        assert float((a - c).abs().max()) <= float(a.abs().max()) / share


def test_wait_runs_out_and_the_context_stays_usable(monkeypatch):
    """One ring slot of every run is left out: the MMA warps' waits run out, then those for the tiles that were never
    finished; nothing hangs, and the next forward is right without anybody asking for the status in between."""
    monkeypatch.setenv("CS_WAIT_LIMIT_US", "2000")
    monkeypatch.setenv("CS_CHAIN", "1")
    cfg = CONFIGS["wide"]
    ctx, _ = make_pair(cfg, 128, 1, 10)
    kv0 = inputs.synthetic_kv(cfg, 1, 128, 100, seed=3, device="cuda")
    tok = i32(np.random.default_rng(0).integers(0, cfg.vocab, size=(1, 11)))

    def step():
        kv, logits = kv0.clone(), torch.zeros(1, 11, cfg.vocab, dtype=torch.float32, device="cuda")
        ctx.cs_verify_step(tok[:, 0].contiguous(), tok[:, 1:].contiguous(), i32([10]), kv, i32([100]), logits_dbg=logits)
        return kv, logits

    want = step()
    assert ctx.cs_sync_status() == cs.CS_OK
    for unit in (0, 2):
        for ask in (True, False):
            ctx.cs_debug_drop_chain_tile(unit)
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            step()
            ev[1].record()
            torch.cuda.synchronize()
            assert 1.0 <= ev[0].elapsed_time(ev[1]) <= 500.0
            if ask:
                assert ctx.cs_sync_status() == cs.CS_ERR_TIMEOUT
            got = step()
            assert ctx.cs_sync_status() == (cs.CS_OK if ask else cs.CS_ERR_TIMEOUT)
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert ctx.workspace_guards_intact()
    ctx.close()


# what decides whether a block is chained: MiB of a layer's weights, head size, QKV features against model features
RULE = {"89": (_cfg(2048, 16, 4, 128, 5888, layers=1), 0), "98": (_cfg(2048, 16, 4, 128, 6656, layers=1), 8),
        "98, QKV of 3 d": (_cfg(2048, 16, 16, 128, 5632, layers=1), 0), "108, heads of 64": (_cfg(2048, 32, 8, 64, 7488, layers=1), 0),
        "116, heads of 64": (_cfg(2048, 32, 8, 64, 8192, layers=1), 8), "135": (_cfg(2560, 20, 4, 128, 7168, layers=1), 12),
        "191": (_cfg(3072, 24, 8, 128, 8128, layers=1), 12), "192": (_cfg(3072, 24, 8, 128, 8192, layers=1), 32),
        "198, QKV of 3 d": (_cfg(3072, 24, 24, 128, 7168, layers=1), 24), "195, heads of 64": (_cfg(3072, 48, 8, 64, 8704, layers=1), 12),
        "245, narrow": (_cfg(2048, 16, 4, 128, 19200, layers=1), 16), "288, heads of 64": (_cfg(4096, 64, 8, 64, 9216, layers=1), 32)}


ROWS = (1, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33)


@pytest.mark.parametrize("name", list(RULE))
def test_blocks_are_chained_where_that_was_measured_to_gain(name, monkeypatch):
    """Three launches a layer where the block is chained, six where it is not."""
    monkeypatch.delenv("CS_CHAIN", raising=False)
    cfg, most = RULE[name]
    ctx = cs.Context(cfg, inputs.make_weights(cfg, seed=4, device="cuda"), max_seq=64, max_batch=1, k_max=32)
    launches = []
    for rows in ROWS:
        hd, ld, kvl = i32(np.zeros((1, 64))), i32([8]), i32([7])
        ctx.cs_loop_begin(hd, ld, ctx.alloc_kv(), kvl, 3, rows - 1, 4)
        launches.append((rows, ctx.cs_loop_launches_per_step()))
        ctx.cs_loop_end()
    ctx.close()
    most_launches = max(n for _, n in launches)
    assert [rows for rows, n in launches if n == most_launches - 3] == [r for r in ROWS if r <= most]
    assert {n for _, n in launches} <= {most_launches, most_launches - 3}
