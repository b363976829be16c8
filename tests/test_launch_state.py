"""What a launch keeps on the device between calls, checked in the source: two launches that share a word by accident can hand out wrong
offsets and write outside their outputs, so the fault itself is never run."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_22441_b200", "csrc")


def _function(file, head):
    """The body behind `head`, without comments and without what only the bounds-checked build compiles."""
    src = open(os.path.join(CSRC, file)).read()
    at = src.index("{", src.index(head))
    depth, i = 1, at + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    body = re.sub(r"//[^\n]*", "", src[at:i])
    return re.sub(r"#ifdef CCR_DEBUG_BOUNDS.*?(#else(.*?))?#endif", lambda m: m.group(2) or "", body, flags=re.S)


def test_compaction_keeps_no_state_in_the_store():
    """A captured call would keep a word of the store's for ever, while direct calls take the same word in turn."""
    body = _function("ccr_api.cu", "ccr_status ccr_compact_valid(")
    assert body.count("launch_chained(") == 2
    assert "status" not in body.replace("ccr_status", "") and "kSchedRegions" not in body
    assert "atomic" not in _function("ccr_pad.cuh", "count_valid_kernel(") + _function("ccr_pad.cuh", "compact_valid_kernel(")


def test_pads_let_only_the_join_of_their_call_start_early():
    """What follows the pads of a call without a join may read them: it is ordered behind their last store."""
    kernel = _function("ccr_pad.cuh", "pad_fill_kernel(")
    assert kernel.index("pdl_wait();") < kernel.index("if (join_follows) pdl_trigger();") and kernel.count("pdl_trigger") == 1
    join, padded = _function("ccr_api.cu", "ccr_status join_impl("), _function("ccr_api.cu", "ccr_status padded_impl(")
    assert "launch_pads(" in padded and ", false)" in padded[padded.index("launch_pads("):]
    at = join.index("launch_pads(")
    assert ", true)" in join[at:] and "CCR_ERR_INVALID_ARG" not in join[at:] and "CCR_ERR_UNSUPPORTED" not in join[at:]
