"""cs_step_host behind a call that failed on its way (its stream was being captured, so that nothing of it
ran): the same call made again brings everything to the device that the failed one had only meant to."""
import ctypes as C
import glob
import os

import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs, inputs

pytestmark = pytest.mark.gpu


def test_a_step_made_again_after_a_failed_one():
    rt = C.CDLL(glob.glob(os.path.join(os.path.dirname(torch.__file__), "..", "nvidia", "cuda_runtime", "lib", "libcudart.so.*"))[0])
    cfg, k, n0, stride = inputs.TINY, 4, 60, 128
    ctx = cs.Context(cfg, inputs.weights_to(inputs.make_weights(cfg, seed=2), "cuda"), max_seq=stride, max_batch=1, k_max=k)
    h = np.zeros((1, stride), dtype=np.int32)
    h[0, :n0] = np.random.default_rng(1).integers(0, 30, size=n0)
    hist, lens = torch.from_numpy(h).pin_memory(), torch.full((1,), n0, dtype=torch.int32).pin_memory()
    hist_d, len_d = torch.zeros(1, stride, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    kv, kvl = ctx.alloc_kv(), torch.full((1,), n0 - 1, dtype=torch.int32, device="cuda")
    acc, out = torch.zeros(1, dtype=torch.int32).pin_memory(), torch.zeros(1, k + 1, dtype=torch.int32).pin_memory()

    def step():
        ctx.cs_step_host(hist, lens, hist_d, len_d, kv, kvl, 3, k, acc, out)

    step()
    for _ in range(2):
        before = int(lens[0])
        torch.cuda.synchronize()
        side, graph = torch.cuda.Stream(), C.c_void_p()
        with torch.cuda.stream(side):
            # (by the runtime: torch's own capture object keeps torch's random numbers captured when its end fails)
            assert rt.cudaStreamBeginCapture(C.c_void_p(side.cuda_stream), 2) == 0          # relaxed
            with pytest.raises(cs.CsError) as err:
                step()
            assert err.value.code == cs.CS_ERR_CUDA
            assert rt.cudaStreamEndCapture(C.c_void_p(side.cuda_stream), C.byref(graph)) != 0 and not graph.value   # the call's look at the stream ended it
            rt.cudaGetLastError()
        torch.cuda.synchronize()
        assert int(lens[0]) == before
        step()
        assert int(lens[0]) == before + int(acc[0]) + 1
        assert hist_d[0, :before].cpu().tolist() == hist[0, :before].tolist() and int(len_d[0]) == before
    assert ctx.cs_sync_status() == cs.CS_OK
    ctx.close()
