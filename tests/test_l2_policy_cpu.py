"""Which loads leave L2 first, read in the source.  Weights do, in the chained and the tall projections; keys and values
that the attention between them left at normal priority would then keep the whole of L2 (8 x 4 rows over 8,000 keys of
the 8B shape: attention 45 -> 51 us a layer, the merge behind it 3 -> 7)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_08923_b200", "csrc")


@pytest.mark.parametrize("source", ["cs_attn_tc.cu", "cs_attn_tcw.cu"])
def test_keys_and_values_leave_l2_first(source):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    loads = re.findall(r"\b(tma_load_2d\w*)\([^;]*&tmKV[^;]*;", text)
    assert loads and set(loads) == {"tma_load_2d_hint"}
