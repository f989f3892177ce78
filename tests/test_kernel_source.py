"""Rules of the device code that can be checked in its source (no GPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_17942_b200", "csrc")


def _calls(text, name):
    """(start, end) of every call of `name`, arguments included."""
    for m in re.finditer(r"\b" + name + r"\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield m.start(), i


def test_issuing_warps_leave_every_wait_together():
    """A warp that walks its loop as a whole while one lane issues: a lane left behind at a wait for two phases of the barrier
    would wait for a parity that is not coming, so every wait's answer is the warp's (__all_sync)."""
    loops = waits = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        for m in re.finditer(r"= elect_lane\(\);", text):
            role = text[m.end():text.index("\n    } else", m.end())]
            together = list(_calls(role, "__all_sync"))
            for beg, end in _calls(role, "mbar_wait"):
                assert any(b < beg and end <= e for b, e in together), f"{os.path.basename(path)}: {role[beg:end]}"
                waits += 1
            loops += 1
    assert loops == 5 and waits >= 2 * loops
