"""The search at the ends of the caller's rows, which need not begin or end on 16 bytes: there a group of four tokens is read token by token.  Rows of every
small length at every offset in a larger buffer, whose other tokens would go on with a match, against the oracle's scan."""
import numpy as np
import pytest

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs
from helpers import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 2, 3])
@pytest.mark.parametrize("tokens", ["constant", "alphabet"])
def test_rows_anywhere_in_a_buffer(tokens, B):
    rng = np.random.default_rng(B)
    for stride in (*range(2, 20), 4095, 4099, 8194):
        for off in range(4):
            buf = np.full(8 + B * stride + 8, 7, np.int32) if tokens == "constant" else rng.integers(0, 3, size=8 + B * stride + 8).astype(np.int32)
            dev = i32(buf)
            hist = buf[off:off + B * stride].reshape(B, stride)
            for gamma in (1, 2, 5, 6):
                lens = [max(0, stride - b) for b in range(B)]
                for policy in (cs.LATEST, cs.FIRST):
                    pos, draft, dlen = (t.cpu().numpy() for t in cs.cs_find_match(dev[off:off + B * stride].view(B, stride), i32(lens), gamma, 5, policy))
                    for b, n in enumerate(lens):
                        p = O.find_match(hist[b], n, gamma, policy)
                        want = O.gather_draft(hist[b], n, p, gamma, 5)
                        assert (int(pos[b]), int(dlen[b]), draft[b].tolist()) == (p, len(want), want + [-1] * (5 - len(want))), (stride, off, gamma, policy, b)
            assert np.array_equal(dev.cpu().numpy(), buf)
