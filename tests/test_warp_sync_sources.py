"""Warp synchronisation in the kernel sources.  __activemask() names the lanes
that happen to be converged, not those that exchange data: a __syncwarp of it
orders nothing between lanes that a branch has parted.  Exchanges through
shared memory name their lanes (or the whole warp) instead."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_12703_gb300", "csrc")


def test_no_synchronisation_of_the_active_lanes():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        assert "__activemask" not in code, name
