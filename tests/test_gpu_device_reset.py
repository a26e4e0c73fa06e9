"""A process that destroys its contexts, resets its device and starts again gets working contexts: nothing
that belonged to the old ones is used.  Runs in a process of its own, without torch's device memory."""
import ctypes as C
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _main():
    import torch
    from paper_2502_08923_b200 import binding as cs, inputs
    lib = cs.load()
    rt = C.CDLL(glob.glob(os.path.join(os.path.dirname(torch.__file__), "..", "nvidia", "cuda_runtime", "lib", "libcudart.so.*"))[0])
    cfg = inputs.TINY
    c = cs.CsModelConfig(cfg.n_layers, cfg.d_model, cfg.n_heads, cfg.n_kv_heads, cfg.head_dim, cfg.d_ffn, cfg.vocab, 64, 1, 4,
                         cfg.rope_theta, cfg.rms_eps)
    need = lib.cs_workspace_bytes(C.byref(c))
    for life in range(2):
        ws, weights = C.c_void_p(), C.c_void_p()
        assert rt.cudaMalloc(C.byref(ws), C.c_size_t(need + 1024)) == 0 and rt.cudaMalloc(C.byref(weights), C.c_size_t(64 << 20)) == 0
        cw = cs.CsWeights()
        for name in ("embed", "lm_head", "final_norm"):
            setattr(cw, name, weights.value)
        per_layer = (C.c_void_p * cfg.n_layers)(*[weights.value] * cfg.n_layers)
        for name in ("attn_norm", "wqkv", "wo", "ffn_norm", "w_gate_up", "w_down"):
            setattr(cw, name, C.cast(per_layer, C.POINTER(C.c_void_p)))
        for _ in range(2):
            h = C.c_void_p()
            assert lib.cs_create(C.byref(h), C.byref(c), C.byref(cw), C.c_void_p((ws.value + 1023) // 1024 * 1024), need) == cs.CS_OK, \
                (life, lib.cs_last_error(None))
            assert lib.cs_sync_status(h, None) == cs.CS_OK
            lib.cs_destroy(h)
        assert rt.cudaDeviceReset() == 0      # ends this process's own context, nothing else
    print("both lives ok")


def test_contexts_after_a_reset_of_the_process_device():
    out = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=ROOT, env={**os.environ, "PYTHONPATH": ROOT}, capture_output=True, text=True,
                         timeout=120)
    assert out.returncode == 0 and "both lives ok" in out.stdout, out.stderr[-2000:]


if __name__ == "__main__":
    _main()
