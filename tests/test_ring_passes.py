"""Rings of y and dx whose readers take alternate heads: a wait by parity alone is satisfied by the load two passes back while the one
between is still under way, so a reader also waits until the slot has been given back.  Shown on a model of the barriers, and looked
for in the source: no run shows that a wait is missing."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_19460_b200", "csrc")


class Barrier:
    def __init__(self):
        self.done = 0                      # completed phases

    def passed(self, parity):              # test_wait.parity: the phase of that parity is not the current one
        return (self.done & 1) != parity


def reads_wrong_load(slots, guarded, heads=24, slow=3):
    """Two readers of alternate heads behind one producer; the load of head `slow` lands last of all that can."""
    full, empty = [Barrier() for _ in range(slots)], [Barrier() for _ in range(slots)]
    content, loaded, read, nxt = [None] * slots, 0, set(), [0, 1]
    pending = []                           # loads under way
    for _ in range(2000):
        moved = False
        if loaded < heads and (loaded < slots or empty[loaded % slots].passed((loaded // slots - 1) & 1)):
            pending.append(loaded)
            loaded += 1
            moved = True
        for r in (0, 1):
            h = nxt[r]
            if h >= heads:
                continue
            s, use = h % slots, h // slots
            if guarded and use and not empty[s].passed((use - 1) & 1):
                continue
            if full[s].passed(use & 1):
                if content[s] != h:
                    return True
                read.add(h)
                empty[s].done += 1
                nxt[r] += 2
                moved = True
        fast = [h for h in pending if h != slow]
        land = fast[:1] or (pending if not moved else [])
        for h in land[:1]:
            pending.remove(h)
            content[h % slots] = h
            full[h % slots].done += 1
            moved = True
        if not moved:
            break
    assert len(read) == heads
    return False


@pytest.mark.parametrize("slots", [3, 5, 7])
def test_a_parity_alone_takes_an_older_load(slots):
    assert reads_wrong_load(slots, guarded=False) and not reads_wrong_load(slots, guarded=True)


def test_every_reader_of_the_rings_waits_that_way():
    src = re.sub(r"//.*", "", open(os.path.join(CSRC, "ssd_tc_scan.cu")).read())
    assert len(re.findall(r"mbar_wait\(&full\[", src)) == 1 and len(re.findall(r"mbar_wait\(&xrfull\[", src)) == 1
    for name in ("empty", "xrempty"):
        body = src[src.index("auto wait_full" if name == "empty" else "auto wait_x"):]
        assert re.match(r"[^;]*\{\s*if \(use\) mbar_wait\(&%s\[slot\], \(use - 1\) & 1," % name, body)
