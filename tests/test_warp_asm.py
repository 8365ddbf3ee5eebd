"""Inline assembly that every lane of a warp must execute together may not be
moved or removed by the compiler: each such statement is volatile."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_17390_gb300", "csrc")


def test_warp_collectives_are_volatile():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        text = open(path).read()
        for m in re.finditer(r"\basm\b\s*(volatile\b)?\s*\(\s*((?:\"[^\"]*\"\s*)+)", text):
            if ".sync" in m.group(2):
                found += 1
                assert m.group(1), "%s: %s" % (os.path.basename(path), m.group(2))
    assert found  # the pattern still meets the statements it is for
