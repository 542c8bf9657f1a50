"""Rules of the device code that no run can show broken, checked on its text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1507_02087_gb300", "csrc")


def conditions_around(text, at):
    """The heads of the blocks that hold position `at`, and the start of its own statement."""
    heads, depth, i = [], 0, at
    start = max(text.rfind(c, 0, at) for c in ";{}")
    heads.append(text[start + 1:at])
    while i > 0:
        i -= 1
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth == 0:
                heads.append(text[max(text.rfind(c, 0, i) for c in ";{}") + 1:i])
            else:
                depth -= 1
    return heads


def test_every_lane_waits_for_another_ctas_memory():
    # The acquire of mbar_wait_cluster orders the memory accesses of the lane that waits.  If one lane waits and a shuffle
    # passes the result on, the other lanes' accesses to shared memory are not ordered: a shuffle orders nothing.
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\bmbar_wait_cluster\(", text):
            found += 1
            heads = conditions_around(text, m.start())
            assert not any("lane ==" in h or "elect_one" in h for h in heads), (path, heads[:3])
    assert found
