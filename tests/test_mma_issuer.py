"""Two orders that no test on a GPU can bring about a failure of, read from the sources.

A tcgen05.commit tells of the MMAs that its own thread has issued, and MMAs are issued by the lane elect.sync names: a commit by
lane 0 would be a drain that waits for nothing if that lane is another.  (Reached only where a bounded wait has run out, which
a test on a GPU does not bring about; so the sources are read.)"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_12825_b200", "csrc")


def test_commits_are_made_by_the_issuing_lane():
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        seen += len(re.findall(r"elect_one\(\)\) umma_commit", text))
        bad = re.search(r"if \((?:lane|tid)[^\n;{]*\)\s*(?:umma_commit|\{[^}]*umma_commit)", text)
        assert bad is None, (os.path.basename(path), bad.group(0))
    assert seen >= 4                           # the drains of the four kernels


def test_the_abort_flag_is_set_up_by_the_warp_that_waits_for_nobody():
    """The producer of the wide kernel arrives at the start barrier without waiting there, and reads the flag: it has to be the one that
    clears it, or it could read what the preceding CTA left."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "attend_tc.cu")).read())
    prologue = text[text.index("if (warp == C::PRODUCER_WARP) {"):]
    producer = prologue[:prologue.index("else if (warp == C::MMA_WARP)")]
    assert "bar_start_arrive" in producer and "bar_start_wait" not in producer
    assert producer.index("*abort_flag = aligned") < producer.index("bar_start_arrive")
    assert len(re.findall(r"\*abort_flag = aligned", text)) == 1
