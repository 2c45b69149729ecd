"""Rings of y and dx whose readers take alternate heads: a wait by parity alone is satisfied by the load two passes back while the one
between is still under way, so a reader also waits until the slot has been given back.  Shown on a model of the barriers, and looked
for in the source: no run shows that a wait is missing."""
import os
import random
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


def ring_sizes(mode):
    """Slots of the rings of values, states and (dx) x rows, as the source has them."""
    src = open(os.path.join(CSRC, "ssd_tc_scan.cu")).read()
    dx, y = lambda m: int(m.group(1)), lambda m: int(m.group(2))
    pick = dx if mode == "dx" else y
    sizes = dict((k, pick(re.search(r"int sc_%s\(int mode\) \{ return mode == SC_DX \? (\d+) : (\d+); \}" % k, src))) for k in ("vals", "states"))
    return dict(sizes, x=int(re.search(r"constexpr int SC_XR = (\d+);", src).group(1)))


def turns_of(first, last, hpg):
    """What a CTA's units first .. last - 1 put through the rings, as the kernel's run_at cuts them: per run the columns operand, then its
    heads.  A turn is the number of its head in the CTA, or None for the columns."""
    turns, u, n = [], first, 0
    while u < last:
        run = min(last - u, hpg - u % hpg)
        turns += [None] + list(range(n, n + run))
        u, n = u + run, n + run
    return turns


def farthest(turns, slots, role, columns):
    """The longest way back from one turn of a role to the one before it, in turns (for the first: to one pass ahead of the ring)."""
    mine = [i for i, h in enumerate(turns) if (columns if h is None else h % 2 == role)]
    return max([b - a for a, b in zip(mine, mine[1:])] + [mine[0] - slots + 1] if mine else [0])


@pytest.mark.parametrize("mode", ["y", "dx"])
@pytest.mark.parametrize("hpg", [2, 4, 6, 10, 24, 80])
def test_a_role_sees_every_second_pass_at_least(mode, hpg):
    """A wait until a slot has been given back is right if the role's turn before lies at most the ring's slots back.  All the ways in which
    a CTA's part can begin and end, the columns operand in turns of its own."""
    size = ring_sizes(mode)
    for first in range(hpg):
        for last in range(first + 1, first + 4 * hpg + 1 if hpg < 24 else first + 2 * hpg + 2):
            turns = turns_of(first, last, hpg)
            for role in (0, 1):
                for columns in (False, True):            # the first issuer takes the columns, nobody else
                    if columns and role:
                        continue
                    assert farthest(turns, size["vals"], role, columns) <= size["vals"]
                    assert farthest(turns, size["states"], role, columns) <= size["states"]
            heads = [h for h in turns if h is not None]   # the x rows have no columns operand among them
            assert mode == "y" or max(farthest(heads, size["x"], r, False) for r in (0, 1)) <= size["x"]


def test_odd_groups_would_not_do():
    """With a head per group the columns take every second turn: four from one head of a role to the next, dx's states have three slots."""
    assert farthest(turns_of(0, 9, 1), 3, 0, False) == 4 > ring_sizes("dx")["states"]


def takes_older(turns, slots, guarded, seed):
    """The ring under a random schedule: whether a role takes a load for the one of a later pass.  Loads land in any order."""
    rng = random.Random(seed)
    full, empty, content = [Barrier() for _ in range(slots)], [Barrier() for _ in range(slots)], [None] * slots
    mine = [[i for i, h in enumerate(turns) if (r == 0 if h is None else h % 2 == r)] for r in (0, 1)]
    nxt, loaded, pending, idle = [0, 0], 0, [], 0
    while idle < 60:
        what, moved = rng.choice(["load", "land", 0, 1]), False
        if what == "load":
            if loaded < len(turns) and (loaded < slots or empty[loaded % slots].passed((loaded // slots - 1) & 1)):
                pending.append(loaded)
                loaded, moved = loaded + 1, True
        elif what == "land":
            if pending:
                t = pending.pop(rng.randrange(len(pending)))
                content[t % slots] = t
                full[t % slots].done += 1
                moved = True
        elif nxt[what] < len(mine[what]):
            t = mine[what][nxt[what]]
            s, use = t % slots, t // slots
            if not (guarded and use and not empty[s].passed((use - 1) & 1)) and full[s].passed(use & 1):
                if content[s] != t:
                    return True
                empty[s].done += 1
                nxt[what], moved = nxt[what] + 1, True
        idle = 0 if moved else idle + 1
    assert nxt == [len(mine[0]), len(mine[1])]
    return False


@pytest.mark.parametrize("hpg,first,heads", [(2, 1, 20), (2, 0, 19), (6, 5, 26), (4, 3, 17)])
@pytest.mark.parametrize("mode", ["y", "dx"])
def test_rings_with_columns_turns(mode, hpg, first, heads):
    turns = turns_of(first, first + heads, hpg)
    for slots in ring_sizes(mode).values():
        assert not any(takes_older(turns, slots, True, seed) for seed in range(60))
    if hpg > 2:       # (with two, columns and heads come round with three slots, and a role sees every pass)
        assert any(takes_older(turns, 3, False, seed) for seed in range(400))
