"""The waits of the on-chip kernels between warps and thread blocks, read from their source: every loop that
polls decides by a vote of the whole warp.  Its give-up test (Patience::over) votes over all 32 lanes itself,
so a loop that some lanes could leave before the others would leave that vote with missing lanes, and a
bounded wait without its bound."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_22308_gb300", "csrc",
                   "resident.cu")


def _condition(text, at):
    """The condition of the while loop nearest before position at."""
    start = text.rindex("while (", 0, at) + len("while (")
    depth, end = 1, start
    while depth:
        depth += {"(": 1, ")": -1}.get(text[end], 0)
        end += 1
    return text[start:end - 1]


def test_every_wait_of_the_resident_kernels_is_decided_by_the_whole_warp():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    waits = [m.start() for m in re.finditer(r"\.over\(", text)]
    assert len(waits) >= 4
    for at in waits:
        cond = _condition(text, at)
        assert re.match(r"!?__(any|all)_sync\(kFull,", cond), cond
