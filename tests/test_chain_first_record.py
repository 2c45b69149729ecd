"""Forward chain: its producer loads the first block, waits for the first record and only then loads the others.  Whatever it is late by,
that wait has to end: nothing but the producer's own loads can bring a later phase of a barrier that has gone on without it.  Shown on a
model of the roles, with the barrier that the source names; a late producer cannot be arranged on a GPU."""
import os
import random
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_19460_b200", "csrc", "ssd_tc_chain.cu")


class Barrier:
    def __init__(self):
        self.done = 0                      # completed phases

    def passed(self, parity):              # try_wait.parity: the phase of that parity is not the current one
        return (self.done & 1) != parity


def ends(once, stages, buffers, late, blocks=12, seed=0):
    """Whether every block is summed.  The producer looks for the first record (`once`: on a barrier of its own, else on the first
    buffer's) when the other roles have had `late` turns; a record waits for its buffer, a sum for its block and its record."""
    rng = random.Random(seed)
    vfull, vempty = [Barrier() for _ in range(buffers)], [Barrier() for _ in range(buffers)]
    first = Barrier() if once else vfull[0]
    loaded, records, summed, go, turns = 1, [0, 1], 0, False, 0
    idle = 0
    while idle < 50:
        role, moved = rng.choice(["producer", "record0", "record1", "sum"]), False
        if role == "producer":
            if not go:
                go = moved = turns >= late and first.passed(0)
            elif loaded < blocks and loaded - summed < stages:
                loaded += 1
                moved = True
        elif role == "sum":
            buf = summed % buffers
            if summed < loaded and vfull[buf].passed(summed // buffers & 1):
                vempty[buf].done += 1
                summed += 1
                moved = True
        else:
            w = int(role[-1])              # records alternate between two warps
            i = records[w]
            buf = i % buffers
            if i < blocks and (i < buffers or vempty[buf].passed(i // buffers - 1 & 1)):
                vfull[buf].done += 1
                first.done += once and i == 0
                records[w] += 2
                moved = True
        turns += role != "producer"
        idle = 0 if moved else idle + (turns >= late)
    return summed == blocks


@pytest.mark.parametrize("stages,buffers", [(4, 4), (3, 2)])          # one head per CTA, two
def test_a_late_producer_goes_on(stages, buffers):
    src = re.sub(r"//.*", "", open(SRC).read())
    name = re.search(r"!BWD && i == 1\) mbar_wait\((\w+), 0,", src).group(1)
    # a barrier that a record arrives on only once, or the first buffer's, on which every so many blocks one does
    once = name != "vfull" and re.search(r"if \(i == 0 && hl == 0\) mbar_arrive\(%s\)" % name, src) is not None
    for late in range(0, 40, 4):
        for seed in range(20):
            assert ends(once, stages, buffers, late, seed=seed), (late, seed)
    # the first buffer's is no such barrier: late enough, the wait is for a phase that cannot come
    assert not all(ends(False, stages, buffers, 36, seed=s) for s in range(20))
