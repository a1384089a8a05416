"""Memory order that no run on one chip can show: read from the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_08814_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _after_waits(code):
    """What follows each shuffle that passes on the outcome of one lane's barrier wait, up to the next statements."""
    for m in re.finditer(r"\w+ = mbar_wait_\w+\(", code):
        line = code[code.rfind("\n", 0, m.start()) + 1:m.start()]
        if not re.search(r"== 0\)\s*$", line):  # the wait of one lane, in an if of its own
            continue
        rest = code[m.end():]
        shuffle = re.search(r"__shfl_sync\(", rest)
        yield rest[shuffle.end():].split("\n")[1:2] if shuffle else [""]


def test_a_wait_by_one_lane_orders_memory_for_its_warp():
    # __shfl_sync converges the lanes but orders no memory among them: a __syncwarp has to follow before the other lanes
    # touch what the barrier guards
    found = 0
    for name in sorted(os.listdir(CSRC)):
        for nxt in _after_waits(_code(name)):
            found += 1
            assert nxt and nxt[0].strip() == "__syncwarp();", (name, nxt)
    assert found >= 1


def test_a_wait_that_ran_out_is_repeated_on_its_own_phase():
    # after a timeout the inference kernel waits once more for the MMAs it issued; on the next phase's parity that wait would
    # return at once and tensor memory be freed under them
    code = _code("mlp.cu")
    waits = re.findall(r"ok = __syncthreads_and\(done\) != 0;\s*(.*?)\n\s*(.*?)\n", code)
    assert waits == [("if (!ok) break;", "phase ^= 1u;")] * 2, waits
