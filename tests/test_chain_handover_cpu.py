"""What one run of the chained projections hands to another, read in the source: what the memory model promises about an
access cannot be made to fail on a GPU at will."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_08923_b200", "csrc")


def _function(name):
    """Body of a device function of the chained projections, without comments."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "cs_chain.cu")).read())
    at = re.search(rf"\b{name}\s*\([^;{{]*\)\s*\{{", text).end()
    depth, end = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
    return text[at:end].replace("\\n", "\n")


def test_a_sum_and_its_mark_are_one_element_of_the_access():
    # a vector access is one access per element, in no stated order: a mark tells of its own element only
    for name, kind in (("put_pair", "st"), ("peek_pair", "ld")):
        accesses = re.findall(r"\b(ld|st)\.[\w.]*global[\w.]*", _function(name))
        assert accesses == [kind], name
        assert re.search(rf"\b{kind}\.[\w.]*global\.v2\.b64\b", _function(name)), name


def test_a_poll_by_a_warp_orders_memory_for_all_its_lanes():
    # the lane whose word it was has acquired it; a vote says so to the others but orders nothing for them
    body = _function("poll_words")
    assert "ld_acquire" in body and re.search(r"__ballot_sync.*__syncwarp\(\);\s*return got;", body, flags=re.S)
