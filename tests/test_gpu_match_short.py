"""Short histories in long rows: the CTAs of a cluster have few candidates each or none, and rows begin anywhere within 16 bytes.  Every length
from 0 to 260 at every such offset, against the oracle's scan; behind a row's length lie tokens that would go on with a match."""
import numpy as np
import pytest

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs
from helpers import i32

pytestmark = pytest.mark.gpu

LONGEST = 260


def _histories(tokens, stride):
    """[4 * (LONGEST + 1)][stride] and the lengths: each of them in four neighbouring rows, which begin at the offsets that the stride gives."""
    lens = np.repeat(np.arange(LONGEST + 1, dtype=np.int32), 4)
    wide = 2 * LONGEST
    rng = np.random.default_rng(stride)
    if tokens == "distinct":
        rows = np.tile(np.arange(1, wide + 1, dtype=np.int32), (len(lens), 1))
    elif tokens == "constant":
        rows = np.full((len(lens), wide), 7, dtype=np.int32)
    else:
        rows = rng.integers(0, 3, size=(len(lens), wide), dtype=np.int32)
    hist = np.zeros((len(lens), stride), dtype=np.int32)
    for b, n in enumerate(lens):
        hist[b, :wide] = rows[b]
        if tokens == "distinct" and b % 8 >= 4:          # the key again, behind the length and across it
            hist[b, n:2 * n] = hist[b, :n]
    return hist, lens


@pytest.mark.parametrize("tokens", ["distinct", "constant", "alphabet"])
@pytest.mark.parametrize("stride", [4097, 4098, 9001, 9002, 20001, 20003])
def test_short_histories_in_long_rows(stride, tokens):
    hist, lens = _histories(tokens, stride)
    hd, ld = i32(hist), i32(lens)
    for gamma in range(1, 7):
        for policy in (cs.LATEST, cs.FIRST):
            pos, draft, dlen = (t.cpu().numpy() for t in cs.cs_find_match(hd, ld, gamma, 7, policy))
            for b, n in enumerate(lens):
                row = hist[b, :max(1, n)]
                p = O.find_match(row, int(n), gamma, policy)
                want = O.gather_draft(row, int(n), p, gamma, 7)
                got = (int(pos[b]), int(dlen[b]), draft[b].tolist())
                assert got == (p, len(want), want + [-1] * (7 - len(want))), (b, int(n), gamma, policy)
