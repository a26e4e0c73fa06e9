"""The search call's native path against the general one: every form of argument that the call takes gives the same tensors on
either, and what is refused is refused alike."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs
from helpers import i32

pytestmark = pytest.mark.gpu


def _both(monkeypatch, *args, **kw):
    """(outcome of the call, outcome without the native path): the three tensors on the host, or the exception."""
    cs.load()
    got = []
    for native in (cs._search, lambda *a: None):
        monkeypatch.setattr(cs, "_search", native)
        try:
            out = cs.cs_find_match(*args, **kw)
            got.append([(tuple(t.shape), t.dtype, t.device, t.is_contiguous(), t.cpu().tolist()) for t in out])
        except Exception as e:
            got.append((type(e), str(e)))
    monkeypatch.undo()
    return got


def _forms():
    h = i32(np.random.default_rng(0).integers(0, 4, size=(3, 400)))
    n = i32([400, 77, 5])
    wide = i32(np.zeros((3, 800)))
    return {
        "plain": (h, n, 3, 10), "first": (h, n, 3, 10, cs.FIRST), "no draft": (h, n, 2, 0), "one": (h[:1], n[:1], 3, 7), "unaligned": (h.view(-1)[1:1 + 3 * 399].view(3, 399), n, 3, 4),
        "column": (h, n.view(3, 1), 3, 4), "numpy k": (h, n, 3, np.int64(6)), "flag": (h, n, True, 4), "empty": (h[:0], n[:0], 3, 4), "longer lengths": (h, i32([400, 77, 5, 9]), 3, 4),
        "strided": (wide[:, ::2], n, 3, 4), "long": (h.long(), n, 3, 4), "host": (h.cpu(), n, 3, 4), "host lengths": (h, n.cpu(), 3, 4), "flat": (h.view(-1), n, 3, 4),
        "gamma 0": (h, n, 0, 4), "gamma 9": (h, n, 9, 4), "policy": (h, n, 3, 4, 2), "negative k": (h, n, 3, -1), "huge k": (h, n, 3, 1 << 40),
    }


@pytest.mark.parametrize("form", list(_forms()) if torch.cuda.is_available() else ["plain"])
def test_native_and_general_path_agree(form, monkeypatch):
    native, general = _both(monkeypatch, *_forms()[form])
    assert native == general


def test_runs_on_the_current_stream():
    h, n = i32(np.zeros((64, 32768))), i32([32768] * 64)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        h.fill_(7)                                   # (in front of the search on its stream only)
        pos, draft, dlen = cs.cs_find_match(h, n, 3, 4)
    side.synchronize()
    assert pos.tolist() == [32768 - 6] * 64 and dlen.tolist() == [3] * 64 and draft[:, :3].eq(7).all()
