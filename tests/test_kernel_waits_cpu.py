"""The kernels' bounded waits, as far as they can be checked without a GPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_0810_1648_gb300", "csrc")


def _statements():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for part in re.split(r"[;{}]", code):
            yield os.path.basename(path), " ".join(part.split())


def test_no_lane_skips_a_vote_of_its_warp():
    """mbar_wait_warp is a vote of all lanes: whether the warp gets that far is
    not left to each lane's own look at a flag that others set meanwhile (a lane
    that saw it would leave the others in the vote)."""
    calls = [(f, s) for f, s in _statements() if "mbar_wait_warp(" in s and "bool mbar_wait_warp" not in s]
    assert len(calls) > 10
    for f, s in calls:
        before = s[: s.index("mbar_wait_warp(")]
        assert "volatile" not in before and "abort_flag" not in before, (f, s)
