"""The search where a CTA of the cluster has more candidates than its threads hold at a time (4,096): the key planted at the edges of the
CTAs' shares, of a round and of a thread's four, against the oracle's scan."""
import numpy as np
import pytest

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs
from helpers import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [cs.LATEST, cs.FIRST])
@pytest.mark.parametrize("gamma", [1, 5, 6])
@pytest.mark.parametrize("n", [32769, 40003, 70001])
def test_key_at_the_edges(n, gamma, policy):
    share = ((n - 2 * gamma + 1 + 7) // 8 + 3) & ~3
    at = sorted({p for p in (0, 3, 4, 1023, 4095, 4096, share - 1, share, share + 4095, 7 * share + 4096, n - 2 * gamma) if 0 <= p <= n - 2 * gamma})
    hist = np.tile(np.arange(1, n + 1, dtype=np.int32), (len(at) + 1, 1))      # the last row has no match
    for b, p in enumerate(at):
        hist[b, p:p + gamma] = hist[b, n - gamma:]
    pos, draft, dlen = cs.cs_find_match(i32(hist), i32([n] * len(hist)), gamma, 7, policy)
    for b, row in enumerate(hist):
        p = O.find_match(row, n, gamma, policy)
        want = O.gather_draft(row, n, p, gamma, 7)
        assert pos[b].item() == p and draft[b].tolist() == want + [-1] * (7 - len(want)) and dlen[b].item() == len(want)
