"""The block kernel's decisions that all warps of a CTA take alike (leave the stage
loop, or go on to the last walkers) and its barriers, on the CPU.

A warp that leaves passes one barrier less than one that goes on, so every warp must
take the same decision: the shared words it rests on (nodes in the tree, the sample's
status) have to be read where no other warp can still change them.  The order of the
reads and barriers at the end of the sweeps is taken from the source, and every
interleaving of two warps that follow it is tried: both must pass the same barriers."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_10290_gb300", "csrc",
                      "sampler_block.cu")


def tail_of_stage():
    """Reads of the two words, barriers and the leave decision from the end of the
    sweeps' passes to the end of the stage, in order."""
    with open(SOURCE) as f:
        text = f.read()
    a = text.index("first = false;\n        }\n") + len("first = false;\n        }\n")
    b = text.index("const unsigned st = lds(ctl + cStatus);", a)
    code = "\n".join(line.split("//")[0] for line in text[a:b].splitlines())
    ops = []
    for m in re.finditer(r"group_sync\(\)|lds\(ctl \+ cDone\) >= n|if \((\w+|lds[^;]*)\) break;", code):
        if m.group(0).startswith("group_sync"):
            ops.append("sync")
        elif m.group(0).startswith("if"):
            ops += (["read"] if "lds" in m.group(1) else []) + ["leave"]
        else:
            ops.append("read")
    return ops


def barriers_agree(ops):
    """Whether two warps pass the same number of barriers whatever their speeds.  `ops`
    up to 'leave' run in order; a warp that has read "not complete" walks (and may
    complete the tree) before its next barrier, one that has read "complete" goes
    straight to the last one."""
    cut = ops.index("leave")
    ends = set()

    def step(pc, seen, count, done, waiting):
        # A barrier opens when both warps wait, or the other has ended (a hang if not).
        if all(waiting):
            return step(pc, seen, (count[0] + 1, count[1] + 1), done, (False, False))
        moved = False
        for w in range(2):
            if waiting[w] or pc[w] == "end":
                continue
            moved = True
            put = lambda t, x: (x, t[1]) if w == 0 else (t[0], x)   # noqa: E731
            if pc[w] == "walk":
                step(put(pc, "last"), seen, count, True, waiting)   # completes the tree
            elif pc[w] == "last":                                   # the barrier after the walkers
                step(put(pc, "final"), seen, count, done, put(waiting, True))
            elif pc[w] == "final":                                  # the barrier before the status is read
                step(put(pc, "end"), seen, count, done, put(waiting, True))
            elif pc[w] == cut:
                step(put(pc, "final" if seen[w] else "walk"), seen, count, done, waiting)
            elif ops[pc[w]] == "read":
                step(put(pc, pc[w] + 1), put(seen, done), count, done, waiting)
            else:
                step(put(pc, pc[w] + 1), seen, count, done, put(waiting, True))
        if not moved:
            ends.add(not any(waiting))
        return None

    step((0, 0), (False, False), (0, 0), False, (False, False))
    return ends == {True}


def test_warps_leave_the_stage_together():
    assert barriers_agree(tail_of_stage())


@pytest.mark.parametrize("ops,same", [(["read", "sync", "leave"], True), (["sync", "read", "leave"], False)])
def test_the_model_tells_the_orders_apart(ops, same):
    assert barriers_agree(ops) == same
