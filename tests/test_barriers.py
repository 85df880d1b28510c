"""Named barriers in the kernels' source: a bar.sync is for whole warps, so the
lanes have to be brought together right before each, whatever ran before it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_05535_gb300", "csrc")


def test_every_named_barrier_follows_a_warp_reconvergence():
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"asm volatile\(\"bar(?:rier)?\.(?:cta\.)?sync", code):
            seen += 1
            assert re.search(r"__syncwarp\(\);\s*$", code[:m.start()]), (path, code[m.start():m.start() + 60])
    assert seen  # the pairing's search barrier
