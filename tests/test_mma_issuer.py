"""A tcgen05.commit tells of the MMAs that its own thread has issued, and MMAs are issued by the lane elect.sync names: a commit by
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
