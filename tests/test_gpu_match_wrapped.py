"""The search call inside a transform that hands in tensors without memory of their own: refused with the general path's error, and the next call works."""
import numpy as np
import pytest
import torch

from paper_2502_08923_b200 import binding as cs
from helpers import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", ["both", "history", "lengths"])
def test_inside_vmap(batched, monkeypatch):
    hist, n = i32(np.full((2, 3, 400), 7)), i32(np.full((2, 3), 400))
    dims = {"both": (0, 0), "history": (0, None), "lengths": (None, 0)}[batched]
    args = tuple(t if d == 0 else t[0] for t, d in zip((hist, n), dims))
    call = torch.vmap(lambda a, b: cs.cs_find_match(a, b, 3, 4), in_dims=dims)
    cs.load()
    said = []
    for native in (cs._search, lambda *a: None):
        monkeypatch.setattr(cs, "_search", native)
        with pytest.raises(RuntimeError) as e:
            call(*args)
        said.append(str(e.value))
    assert said[0] == said[1]
    monkeypatch.undo()
    pos, _, dlen = cs.cs_find_match(hist[0], n[0], 3, 4)
    assert pos.tolist() == [394] * 3 and dlen.tolist() == [3] * 3
