"""Rules of the device code that no run can show broken, checked on its text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1507_02087_gb300", "csrc")


def waits_passed_on_by_a_shuffle():
    """(file, the statements after it) of each cluster-scope barrier wait of one lane, result passed on by a shuffle."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\bmbar_wait_cluster\(", text):
            after = text[m.end():]
            shfl = re.search(r"= __shfl_sync\([^;]*;", after)
            assert shfl, path
            found.append((os.path.basename(path), after[shfl.end():shfl.end() + 200].strip()))
    return found


def test_a_wait_by_one_lane_orders_the_memory_of_the_others():
    # The acquire of mbar_wait_cluster orders the memory accesses of the lane that waits.  A shuffle passes its result
    # on but orders nothing, so the other lanes' accesses to shared memory need a __syncwarp first.
    found = waits_passed_on_by_a_shuffle()
    assert found
    for name, rest in found:
        assert rest.startswith("__syncwarp();"), (name, rest)
