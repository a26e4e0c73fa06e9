"""The pipelined tcgen05 attention kernel (query rows as M) at the sizes where it can go wrong: key
ranges around its 128-key tiles, slices of one, two and more tiles than its ring of six slots holds,
blocks at the edges of its 32-lane quarters and its 128-row groups, sequences whose rows are shorter
than the longest of the batch; and the choice between it and the kernel with the keys as M on both
sides of the line.  Against the mma.sync kernel on the same inputs.

Tolerance: queries and weights are two bf16 terms in every kernel (relative 2^-17 per factor) and sums
are fp32, so the first layer agrees to about 2^-15; a K or V element of the second layer that this
moves across a rounding boundary of bf16 differs by 2^-8 of itself and is one of many keys, so no logit
can move by more than 2^-8 of the largest."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu

CFG = inputs.ModelConfig(n_layers=2, d_model=256, n_heads=8, n_kv_heads=2, head_dim=128, d_ffn=512,
                         vocab=512, rope_theta=500000.0, rms_eps=1e-5)


@pytest.fixture(scope="module")
def weights():
    return inputs.weights_to(inputs.make_weights(CFG, seed=12, gain_jitter=0.05), "cuda")


def logits_of(weights, kern, B, k, kv_lens, max_seq, monkeypatch):
    if kern is None:
        monkeypatch.delenv("CS_ATTN_KERNEL", raising=False)
    else:
        monkeypatch.setenv("CS_ATTN_KERNEL", kern)
    rng = np.random.default_rng(k + sum(kv_lens))
    last = rng.integers(0, CFG.vocab, size=B)
    draft = rng.integers(0, CFG.vocab, size=(B, k))
    kv, kvl = inputs.synthetic_kv(CFG, B, max_seq, max(kv_lens), seed=k, device="cuda"), i32(kv_lens)
    ctx = cs.Context(CFG, weights, max_seq=max_seq, max_batch=B, k_max=max(k, 1))
    logits = torch.full((B, k + 1, CFG.vocab), float("nan"), dtype=torch.float32, device="cuda")
    dr = i32(draft) if k > 0 else torch.zeros((B, 0), dtype=torch.int32, device="cuda")
    ctx.cs_verify_step(i32(last), dr, i32([k] * B), kv, kvl, logits_dbg=logits)
    assert ctx.cs_sync_status() == 0
    out = logits.cpu().numpy()
    ctx.close()
    return out


@pytest.mark.parametrize("B,k,kv_lens", [
    (1, 0, [127]), (1, 0, [128]), (1, 0, [129]),               # one row, around one tile
    (1, 7, [247]), (1, 7, [249]),                              # 32 query rows: one lane quarter; two and three tiles
    (1, 8, [1023]),                                            # 33rd query row
    (1, 31, [4096]), (1, 32, [4097]),                          # 128 query rows, and two row groups
    (1, 100, [6000]), (2, 60, [9000, 300]),                    # several groups, several tiles a slice
    (16, 10, [6000, 1] + [128 * i + 5 for i in range(14)]),    # four slices of up to twelve tiles, the ring wraps
    (16, 0, [5000] + [640] * 15),
])
def test_rows_as_m_agrees_at_the_edges(weights, B, k, kv_lens, monkeypatch):
    max_seq = max(kv_lens) + k + 9
    ref = logits_of(weights, "mma", B, k, kv_lens, max_seq, monkeypatch)
    got = logits_of(weights, "tc", B, k, kv_lens, max_seq, monkeypatch)
    assert np.isfinite(got).all()
    assert float(np.abs(got - ref).max()) < 2.0 ** -8 * float(np.abs(ref).max())


@pytest.mark.parametrize("k", [11, 12])
@pytest.mark.parametrize("tiles", [80, 84])
def test_choice_between_the_tcgen05_kernels(weights, k, tiles, monkeypatch):
    """12 and 13 block rows (48 and 52 query rows), 20 and 21 tiles for each of the four slices."""
    B, max_seq = 16, tiles * 128
    kv_lens = [max_seq - k - 1 - 40 * b for b in range(B)]
    ref = logits_of(weights, "mma", B, k, kv_lens, max_seq, monkeypatch)
    got = logits_of(weights, None, B, k, kv_lens, max_seq, monkeypatch)
    assert np.isfinite(got).all()
    assert float(np.abs(got - ref).max()) < 2.0 ** -8 * float(np.abs(ref).max())
