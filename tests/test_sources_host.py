"""No kernel or launcher counts on a number of SMs: grids and dispatch rules take the device's."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_10711_b200", "csrc")


def test_the_sm_count_is_a_literal_in_one_place():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        with open(path) as f:
            for line in f:
                code = re.sub(r"//.*", "", line)
                if re.search(r"\b148l?\b", code):
                    found.append((os.path.basename(path), code.strip()))
    assert found == [("wino_launch.h", "constexpr int kDefaultSms = 148;")]
