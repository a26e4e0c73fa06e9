"""A generation call gives back what it took: contexts that have run loops long enough to capture a
step hold no more device memory than contexts that have not."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs

pytestmark = pytest.mark.gpu


def test_long_loops_leave_no_device_memory_behind():
    cfg = inputs.ModelConfig(n_layers=12, d_model=2048, n_heads=16, n_kv_heads=4, head_dim=128, d_ffn=4096, vocab=2000,
                             rope_theta=500000.0, rms_eps=1e-5)
    w = inputs.make_weights(cfg, seed=6, device="cuda")
    ctxs = [cs.Context(cfg, w, max_seq=200, max_batch=1, k_max=1) for _ in range(20)]
    kv = ctxs[0].alloc_kv()
    hist = torch.from_numpy(np.random.default_rng(1).integers(0, 60, size=(1, 200)).astype(np.int32)).cuda()

    def run(ctx, new):
        hl = torch.tensor([100], dtype=torch.int32, device="cuda")
        ctx.cs_decode_loop(hist.clone(), hl, kv, hl - 1, 3, 1, new)

    run(ctxs[0], 12)                     # the first capture of a process takes memory for the runtime
    for ctx in ctxs:
        run(ctx, 3)                      # enqueued step by step
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for ctx in ctxs:
        run(ctx, 12)                     # captured: 20 graphs that stay take 6 MB
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free
    for ctx in ctxs:
        ctx.close()
