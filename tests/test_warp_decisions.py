"""Decisions that a warp takes on a word which other threads change are taken
once for the warp.  Lanes that load such a word for themselves may see different
values; full-mask operations after the branch then wait for lanes that have gone
another way, without a limit.  Checked in the sources: no run can show it safely."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1112_0059_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_hand_over_words_are_read_under_a_vote():
    text = _source("knn_tc.cu")
    loads = [m.start() for m in re.finditer(r"ld_shared_acquire\(", text)]
    assert len(loads) >= 3  # the inserter's poll, the epilogue's check and its wait
    for at in loads:
        before = re.split(r"[;{}]", text[:at])[-1]
        assert re.search(r"__(all|any)_sync\(0xffffffffu,\s*$", before), text[at - 80:at + 60]


def test_error_word_is_read_by_one_thread():
    text = _source("knn_tc.cu")
    reads = [m.start() for m in re.finditer(r"volatile uint32_t\*>\(dev_err\)", text)]
    assert len(reads) == 1
    opened = text[:reads[0]].rindex("if (threadIdx.x == 0) {")
    assert "}" not in text[opened:reads[0]]  # inside that branch; the CTA reads what it stored after the barrier
