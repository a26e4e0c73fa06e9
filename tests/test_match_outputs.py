"""What cs_find_match and the index's lookup return when the caller gives no outputs: [B], [B][k], [B] for
the B rows of the history, however many lengths come with it; a negative k is the library's error."""
import numpy as np
import pytest
import torch

from oracle import copyspec_oracle as O
from paper_2502_08923_b200 import binding as cs


@pytest.mark.parametrize("B,k", [(1, 10), (3, 4), (2, 0), (2, -1)])
def test_shapes_follow_the_history(B, k):
    for lens in ((B,), (B + 3,), (B, 1), (1, B)):
        mp, dr, dl = cs._match_outputs(torch.zeros(B, 16, dtype=torch.int32), torch.zeros(lens, dtype=torch.int32), k)
        assert mp.shape == dl.shape == (B,) and dr.shape == (B, max(k, 0))
        assert all(t.dtype == torch.int32 and t.is_contiguous() for t in (mp, dr, dl))


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(5,), (2,), (2, 1), (1, 4)])
def test_lengths_of_a_larger_batch(shape):
    rng = np.random.default_rng(3)
    hist = rng.integers(0, 3, size=(2, 64)).astype(np.int32)
    lens = np.zeros(shape, dtype=np.int32)
    lens.reshape(-1)[:2] = (60, 41)
    hd, ld = torch.from_numpy(hist).cuda(), torch.from_numpy(lens).cuda()
    index = cs.GramIndex(2, 64, 3)
    index.cs_gram_index_update(hd, ld)
    for mp, dr, dl in (cs.cs_find_match(hd, ld, 3, 5), index.cs_find_match_indexed(hd, ld, 5)):
        assert mp.shape == dl.shape == (2,) and dr.shape == (2, 5)
        for b, n in enumerate((60, 41)):
            p = O.find_match(hist[b], n, 3, cs.LATEST)
            d = O.gather_draft(hist[b], n, p, 3, 5)
            assert int(mp[b]) == p and int(dl[b]) == len(d) and dr[b, :len(d)].tolist() == [int(t) for t in d]
    with pytest.raises(cs.CsError) as err:
        cs.cs_find_match(hd, ld, 3, -1)
    assert err.value.code == cs.CS_ERR_ARG
