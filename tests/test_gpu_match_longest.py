"""The search over the longest rows that an int counts: positions near 2^31 do not wrap.  Distinct tokens with the key planted at the edges."""
import pytest
import torch

from paper_2502_08923_b200 import binding as cs

pytestmark = pytest.mark.gpu

LONGEST = (1 << 31) - 1


def test_positions_near_the_largest_int():
    row = torch.arange(LONGEST, dtype=torch.int32, device="cuda")
    for n in (LONGEST, LONGEST - 1, LONGEST - 1500, LONGEST - 4097):
        length = torch.tensor([n], dtype=torch.int32, device="cuda")
        for gamma in (1, 5, 6) if n == LONGEST else (1, 5):
            first, last = 4096 * 7 + 3, n - 2 * gamma
            for policy, want in ((cs.LATEST, (-1, last, last)), (cs.FIRST, (-1, last, first))):
                for at, p in zip((None, last, first), want):          # no match, one at the last candidate, another far ahead of it
                    if at is not None:
                        row[at:at + gamma] = row[n - gamma:n]
                    pos, draft, dlen = cs.cs_find_match(row[None], length, gamma, 7, policy)
                    got = 0 if p < 0 else min(7, n - p - gamma)
                    assert (pos.item(), dlen.item()) == (p, got), (n, gamma, policy, at)
                    assert draft[0, :got].tolist() == (row[p + gamma:p + gamma + got].tolist() if got else []) and draft[0, got:].tolist() == [-1] * (7 - got)
                for at in (last, first):
                    row[at:at + gamma] = torch.arange(at, at + gamma, dtype=torch.int32, device="cuda")
