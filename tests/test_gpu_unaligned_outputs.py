"""Output buffers that begin off a 16-byte boundary (a contiguous view behind an odd number of floats):
their contents equal those of an aligned buffer, whether rows are multiples of 16 bytes or not, and the
floats around them are left alone."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import inputs
from helpers import i32, make_pair

pytestmark = pytest.mark.gpu


def _view(off, *shape):
    n = int(np.prod(shape))
    buf = torch.full((n + off + 5,), -7.0, dtype=torch.float32, device="cuda")
    return buf, buf[off:off + n].view(shape)


def _intact(buf, off, n):
    return bool((buf[:off] == -7.0).all() and (buf[off + n:] == -7.0).all())


@pytest.mark.parametrize("vocab", [1000, 1003])
@pytest.mark.parametrize("B,k", [(1, 0), (2, 10), (4, 20)])
def test_logits_anywhere(vocab, B, k):
    cfg = inputs.ModelConfig(n_layers=1, d_model=256, n_heads=2, n_kv_heads=2, head_dim=128, d_ffn=512, vocab=vocab)
    ctx, _ = make_pair(cfg, 64, B, max(k, 1), seed=2)
    rng = np.random.default_rng(1)
    kv0 = inputs.synthetic_kv(cfg, B, 64, 20, seed=3, device="cuda")
    last, draft, dl, script = inputs.verify_inputs_with_tau(rng, B, max(k, 1), rng.integers(0, max(k, 1) + 1, size=B), vocab)
    draft = i32(np.asarray(draft)[:, :k]) if k else None
    dl = i32(np.minimum(dl, k))
    X = torch.randn((B * (k + 1) + 15) // 16 * 16, 256, device="cuda").to(torch.bfloat16)
    got = []
    for off in (0, 1, 2, 3):
        buf, logits = _view(off, B, k + 1, vocab)
        ctx.cs_verify_step(i32(last), draft, dl, kv0.clone(), i32([20 - b for b in range(B)]), logits_dbg=logits)
        head_buf, head = _view(off, B * (k + 1), vocab)
        ctx.cs_lm_head(X, rows=B * (k + 1), logits_dbg=head)
        assert ctx.cs_sync_status() == 0
        assert _intact(buf, off, logits.numel()) and _intact(head_buf, off, head.numel())
        got.append((logits.clone(), head.clone()))
    for pair in got[1:]:
        assert torch.equal(pair[0], got[0][0]) and torch.equal(pair[1], got[0][1])
    ctx.close()


@pytest.mark.parametrize("N", [264, 265])
@pytest.mark.parametrize("rows", [5, 32, 33, 200])     # one-SM tiles up to 32 rows, SM pairs above
def test_linear_output_anywhere(N, rows):
    cfg = inputs.ModelConfig(n_layers=1, d_model=256, n_heads=2, n_kv_heads=2, head_dim=128, d_ffn=512, vocab=512)
    ctx, _ = make_pair(cfg, 64, 1, 10)
    X = torch.randn((rows + 15) // 16 * 16, 2048, device="cuda").to(torch.bfloat16)
    W = torch.randn(N, 2048, device="cuda").to(torch.bfloat16)
    want = ctx.cs_linear(X, W, rows=rows)
    for off in (1, 2, 3):
        buf, Y = _view(off, rows, N)
        ctx._check(ctx.lib.cs_linear(ctx.handle, X.data_ptr(), W.data_ptr(), rows, N, 2048, Y.data_ptr(), torch.cuda.current_stream().cuda_stream), "cs_linear")
        assert ctx.cs_sync_status() == 0 and torch.equal(Y, want) and _intact(buf, off, rows * N)
    ctx.close()
