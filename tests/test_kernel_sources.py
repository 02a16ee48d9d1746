"""Properties of the kernel sources that no run can show (no GPU, no build)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11536_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def text(path):
    """A source without its comments."""
    s = open(path).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_bulk_load_multicasts_to_a_cluster(path):
    """Replicas on several GPUs load this library."""
    s = re.sub(r'"\s*\n?\s*"', "", text(path))  # adjacent literals are one instruction
    for instruction in re.findall(r"cp\.async\.bulk[^;\[]*", s):
        assert ".multicast::cluster" not in instruction, instruction
