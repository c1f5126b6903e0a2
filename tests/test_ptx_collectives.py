"""Inline PTX that a whole warp takes part in (a .sync instruction) is volatile: without that
the compiler may move it, or drop or duplicate it, as it may an arithmetic expression.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2110_08868_gb300", "csrc")


def test_warp_collectives_are_volatile():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = open(path).read()
        for m in re.finditer(r"\basm\b(\s+volatile\b)?\s*\(\s*((?:\"[^\"]*\"\s*)+)", src):
            if ".sync" in m.group(2):
                seen += 1
                assert m.group(1), (os.path.basename(path), m.group(2).strip())
    assert seen >= 2
