"""Hand-written barriers of the CUDA sources: the aligned forms of the PTX
barrier want every lane of a warp at the same instruction, so each follows a
__syncwarp()."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2307_11248_gb300", "csrc")


def test_aligned_barriers_follow_a_syncwarp():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r'asm\s+volatile\s*\(\s*"(?:bar\.sync|barrier(?:\.cta)?\.sync\.aligned)', text):
            seen += 1
            assert re.search(r"__syncwarp\(\);\s*$", text[:m.start()]), (name, text[m.start():m.end()])
    assert seen > 0
