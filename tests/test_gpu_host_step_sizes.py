"""cs_step_host at the ends of what its input and output words hold: one row, 16 sequences of 16
rows (256), 128 of two, with and without a script; histories on the device must be those of the host
after every call, and accepted lengths and tokens (whole numbers) those of the model-free simulator."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs, inputs
from helpers import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,k", [(1, 0), (1, 10), (16, 15), (128, 1), (3, 7)])
def test_scripted_host_steps(B, k):
    cfg = inputs.TINY
    rng = np.random.default_rng(B)
    n0, steps = 60, 4
    max_new = steps * (k + 1) + k + 1
    stride = (n0 + max_new + k + 4) // 4 * 4
    ctx = cs.Context(cfg, inputs.weights_to(inputs.make_weights(cfg, seed=2), "cuda"), max_seq=stride + k, max_batch=B, k_max=max(k, 1))
    ctxts = [rng.integers(0, 40, size=n0).astype(np.int32) for _ in range(B)]       # few ids: matches are frequent
    scripts = [np.concatenate([inputs.copy_script(rng, c, max_new, 0.8, 3, 12, 40, zipf_s=None), np.full(k + 1, -1, np.int32)]) for c in ctxts]
    sims = [O.scripted_simulator(c, s, 3, k, O.LATEST, max_new + k + 1)[0] for c, s in zip(ctxts, scripts)]
    h = np.zeros((B, stride), dtype=np.int32)
    h[:, :n0] = np.stack(ctxts)
    kv, kvl = ctx.alloc_kv(), torch.zeros(B, dtype=torch.int32, device="cuda")
    ctx.cs_prefill(i32(h), i32([n0] * B), n0, kv, kvl)
    hist, lens = torch.from_numpy(h).pin_memory(), torch.full((B,), n0, dtype=torch.int32).pin_memory()
    hist_d, len_d = torch.zeros(B, stride, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    acc, out = torch.zeros(B, dtype=torch.int32), torch.zeros(B, k + 1, dtype=torch.int32)
    for step in range(steps):
        row = np.stack([s[int(lens[b]) - n0:int(lens[b]) - n0 + k + 1] for b, s in enumerate(scripts)])
        before = lens.clone()
        ctx.cs_step_host(hist, lens, hist_d, len_d, kv, kvl, 3, k, acc, out, script_host=torch.from_numpy(row.astype(np.int32)))
        assert len_d.cpu().tolist() == before.tolist()
        for b in range(B):
            rec = sims[b][step]
            assert int(acc[b]) == rec["tau"] and out[b, :rec["tau"] + 1].tolist() == rec["out"], (step, b)
            assert hist_d[b, :int(before[b])].cpu().tolist() == hist[b, :int(before[b])].tolist()
    assert ctx.cs_sync_status() == 0
    assert kvl.cpu().tolist() == [int(x) - 1 for x in lens]
    ctx.close()
