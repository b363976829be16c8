"""Every block of the join kernels waits for the launch in front of it before it leaves, whichever way it leaves: a launch that
completed before its predecessor would let the work behind it start too early.  No wait can be made to run out in a sound launch,
so the exits are checked in the source."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_22441_b200", "csrc")


def _kernel_body(file, name):
    src = open(os.path.join(CSRC, file)).read()
    at = src.index("{", re.search(r"\b%s\(const JoinArgs a" % name, src).start())
    depth, i = 1, at + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return re.sub(r"//[^\n]*", "", src[at:i])


@pytest.mark.parametrize("file,name", [("ccr_join.cuh", "join_kernel"), ("ccr_ws.cuh", "join_ws_kernel")])
def test_no_exit_of_a_join_kernel_without_the_wait(file, name):
    body = _kernel_body(file, name)
    wait = "pdl_wait();"
    if name == "join_kernel":  # the whole block waits in front of its first read
        first = body.index(wait)
        assert not re.search(r"\breturn\b|\bgload\b|\bstage_keys\b", body[:first])
        return
    exits = [m.start() for m in re.finditer(r"\breturn;", body)]
    assert len(exits) == 2  # a block without work, and the streamers
    for e in exits:
        assert body[:e].rstrip().endswith(wait)


def test_document_rows_are_fetched_behind_the_wait():
    """Rows of the store are inputs that the launch in front may have written: an upsert followed by a join on one stream."""
    body = _kernel_body("ccr_ws.cuh", "join_ws_kernel")
    fetch = [m.start() for m in re.finditer(r"\bfetch_docs\(\);", body)]
    assert body[:fetch[0]].rstrip().endswith("pdl_wait();")
    role = body[body.index("if (role_rank >= n_res)"):]
    first = role.index("pdl_wait();")
    assert not re.search(r"\bemit_group\b|\bfetch_docs\(\)", role[:first])  # (the lambda is no call)


def test_inputs_are_read_ahead_only_of_a_join_that_is_still_running():
    """The end of a kernel is no point at which its writes are promised to be visible to a launch that has not waited, so a block looks
    for the ticket of the join in front before it reads anything, and the ticket is there from before the trigger to the block's end."""
    body = _kernel_body("ccr_ws.cuh", "join_ws_kernel")
    settled = body.index("if (__syncthreads_or(in_front) == 0 && may_read_ahead(a)) {")
    behind = body[settled:]
    assert re.match(r"[^}]*\{\s*pdl_wait\(\);\s*if \(n_req_cached > 0\) mirror_offsets\(\);\s*__syncthreads\(\);\s*\}", behind)
    early = body[:settled]
    assert "if (!may_read_ahead(a)) pdl_wait();" in early and early.index("may_read_ahead") < early.index("mirror_offsets();  ".strip())
    # in front of it only the offsets are read, past L1, and they are read again
    assert not re.search(r"\bgload\(|\bstage_keys\b|\ba\.(cand_idx|edge_keys|sched)\s*[+\[]", early)
    assert early.index("show_ticket(a, a.ticket);") > 0
    assert body.count("pdl_trigger()") == 1 and "pdl_trigger()" in behind
    assert body.count("show_ticket(a, 0u);") == len(re.findall(r"\breturn;", body))
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "ccr_api.cu")).read())
    assert "a.behind_pads = n_max > 0 ? 1 : 0;" in src and src.count("behind_pads") == 1


def test_the_look_at_the_next_sub_tile_does_not_wait():
    """A streamer that holds a group must not be held back by a sub-tile that is not there yet."""
    body = _kernel_body("ccr_ws.cuh", "join_ws_kernel")
    assert "if (!block && !__all_sync(kFull, mbar_test_wait(" in body and "mbar_try_wait(" not in body
