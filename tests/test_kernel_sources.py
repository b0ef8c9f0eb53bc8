"""Properties of the kernel sources that hold for the whole library (no GPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_05194_gb300", "csrc")


def code(path):
    src = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)


def test_no_copy_or_commit_goes_to_several_ctas():
    """The library is loaded by every rank of a multi-GPU program: its tile loads and commits
    stay within one CTA."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        assert not re.search(r"multicast", code(path), re.I), os.path.basename(path)
