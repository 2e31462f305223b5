"""Kernel attributes belong to a device: nothing in the library remembers in a
process-wide flag that one was set.  (A second GPU, which would see the
difference, is not needed: the sources are read.)
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1702_04487_gb300", "csrc")


def test_no_process_wide_flags():
    found = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        hits = re.findall(r"\bstatic\s+(?:std::atomic<)?(?:bool|int|unsigned)\b[^;()\n]*[;=]", text)
        if hits:
            found[os.path.basename(path)] = hits
    assert not found, found
