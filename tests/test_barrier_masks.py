"""Warp barriers of the CUDA sources name the lanes they wait for: __activemask() tells which lanes happen to be
converged, which is no promise that the lanes that exchange data are among them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_0330_gb300", "csrc")


def test_no_barrier_or_exchange_takes_its_mask_from_the_converged_lanes():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
    assert files
    for f in files:
        code = re.sub(r"//[^\n]*", "", open(f).read())
        assert not re.search(r"__activemask\s*\(", code), f
