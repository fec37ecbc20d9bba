"""A named barrier (bar.sync) is the aligned form: every lane of a warp has to
reach it together, which after a divergent loop only __syncwarp() ensures."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_named_barriers_follow_a_warp_barrier():
    found = 0
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_1607_03884_gb300", "csrc", "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"asm volatile\(\s*\"bar\.sync", text):
            found += 1
            assert text[:m.start()].rstrip().endswith("__syncwarp();"), (path, text[m.start():][:60])
    assert found >= 2
