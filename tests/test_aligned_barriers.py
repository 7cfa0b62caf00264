"""A cluster barrier's aligned form needs every lane of the warp at the same
instruction: in the source each one comes right after a __syncwarp of its own,
whatever its callers did before."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_22215_gb300", "csrc")


def test_aligned_cluster_barriers_converge_the_warp_first():
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        for m in re.finditer(r'asm volatile\("barrier\.cluster\.[a-z.]*aligned', text):
            found += 1
            assert re.search(r"__syncwarp\(\);\s*$", text[:m.start()]), f"{os.path.basename(path)}: {m.group(0)}"
    assert found >= 2
