"""Hand-written barriers of the CUDA sources: the aligned form of the PTX barrier
wants every lane of a warp at the same instruction, so where the rotation layout's
lanes part before one, a __syncwarp() brings them together."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2307_11248_gb300", "csrc",
                   "qap_rotation.cuh")
# code of some lanes only, or of lanes that leave a loop at different rounds
PARTS = re.compile(r"if \(lane == 0\)|if \(\(threadIdx\.x & 31\) == 0\)|if \(T\.pt == 0\)|rot_update_m<NT|"
                   r"if \(live\[j\]|keeper\.template move|mark\[x\] = 0|d_init\(v0, v1\)")


def _function(text, head):
    start = text.index(head)
    return text[start:text.index("\n}\n", start)]


def test_lanes_meet_before_each_barrier():
    with open(SRC) as f:
        text = re.sub(r"//[^\n]*", lambda m: m.group() if "---- outputs" in m.group() else "", f.read())
    assert len(re.findall(r"bar\.sync", text)) == 1  # rot_barrier() alone
    seen = 0
    for head in ("void rot_clear_marks(", "bool next(int2* red)", "void rot_owner()",
                 "void rot_phase_x()", "void rot_helper()"):
        body = _function(text, head).split("// ---- outputs")[0]
        for m in PARTS.finditer(body):
            after = body[m.end():]
            barrier = after.find("rot_barrier();")
            if head == "bool next(int2* red)":
                barrier = after.index("return")
            assert "__syncwarp();" in (after if barrier < 0 else after[:barrier]), (head, m.group())
            seen += 1
    assert seen >= 8
