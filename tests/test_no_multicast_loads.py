"""The library also serves runs on several GPUs, so no bulk copy in it is a cluster-multicast one (an arrival of
tcgen05.commit on both CTAs' barriers is no copy)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_06344_gb300", "csrc")


def test_no_bulk_copy_is_multicast():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert files
    for f in files:
        with open(f) as fh:
            text = fh.read()
        for m in re.finditer(r"cp\.async\.bulk[^\"\\]*", text):
            assert "multicast" not in m.group(0), (os.path.basename(f), m.group(0))
