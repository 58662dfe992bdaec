"""The resident kernel's warps are whole at its named barriers.

A split warp at an aligned named barrier (bar.sync, bar.arrive) is undefined, and whether a warp
is split there is the compiler's choice, so no run can show the absence of the fault: the source
is checked.  The barriers stand in two functions only, which join the warp themselves except at
the workers' own barrier (1); the poll of the mail boxes, which lanes leave one by one, joins
it before that one."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_13410_gb300", "csrc")


def _code():
    with open(os.path.join(CSRC, "resident.cu")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_named_barriers_join_the_warp():
    code = _code()
    bodies = re.findall(r"void barrier_(?:sync|arrive)\(\) \{(.*?)\n\}", code, flags=re.S)
    assert len(bodies) == 2
    for b in bodies:
        assert re.match(r"\s*if \(ID != 1\) __syncwarp\(\);\s*asm volatile\(\"bar\.", b)
    # no named barrier anywhere else, and barrier 1 only as the workers' sync()
    assert len(re.findall(r"\bbar\.|barrier\.cta", code)) == 2
    assert re.findall(r"barrier_\w+<1,", code) == ["barrier_sync<1,"]


def test_the_poll_joins_the_warp():
    code = _code()
    poll = code[code.index("auto receive = "):code.index("received();", code.index("auto receive = "))]
    assert poll.index("for (;;)") < poll.index("__syncwarp();") < poll.index("w.sync();")
