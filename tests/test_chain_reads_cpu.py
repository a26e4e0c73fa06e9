"""Kernels that start before their predecessor is done (griddepcontrol.wait) must not read words that
other kernels of the chain write through the read-only path: such a kernel may be resident while they
still change, and that path is not coherent across it.  nvcc may take it for any pointer parameter
that is const and __restrict__, so a parameter declared that way is either memory that no kernel
writes, or is never dereferenced directly (only through __ldcg, cp.async or TMA)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_08923_b200", "csrc")
CONSTANTS = {"E", "gain", "inv_freq"}        # embedding, norm gains, rotary frequencies


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s*)?(k_\w+)\s*\((.*?)\)\s*\{", text, flags=re.S):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield f"{os.path.basename(path)}:{m.group(1)}", m.group(2), text[m.end():end]


def _read_directly(body, name):
    # a subscript, or a dereference that no load intrinsic wraps
    return bool(re.search(rf"\b{name}\s*\[", body) or re.search(rf"\*\s*{name}\b", body)
                or re.search(rf"(?<!__ldcg\()\*\s*reinterpret_cast<[^>]*>\(\s*{name}\b", body))


KERNELS = {n: (params, body) for n, params, body in _kernels()}
EARLY = sorted(n for n, (_, body) in KERNELS.items() if "griddepcontrol.wait" in body or "CS_PDL_PROLOGUE" in body)


def test_the_kernels_are_found():
    assert {"cs_layers.cu:k_block_setup", "cs_layers.cu:k_accept", "cs_match.cu:k_find_match", "cs_attn.cu:k_attn_mma",
            "cs_gemm.cu:k_tile_reduce_static", "cs_gemm_pair.cu:k_gemm_pair"} <= set(EARLY)


@pytest.mark.parametrize("kernel", EARLY)
def test_no_chain_word_through_the_read_only_path(kernel):
    params, body = KERNELS[kernel]
    for name in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params):
        assert name in CONSTANTS or not _read_directly(body, name), f"{kernel} reads {name} through a const __restrict__ pointer"
