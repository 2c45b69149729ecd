"""Shared-memory buffers that a bulk or TMA copy refills after ordinary loads have read them: the reads belong to the generic
proxy and the copy to the async proxy, so every role that reads such a buffer has to pass a proxy fence before it gives the
buffer back, or the refill may overtake the read.  Checked in the sources: no run can show that the fence is there."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_19460_b200", "csrc")
FENCED = ("fence_proxy_async_smem()", "tma_store_wait_read()")      # the second: a store has read its source, no load has


def statements(path):
    """The lines of a source file, comments cut off, blank lines left out."""
    lines = (re.sub(r"//.*", "", l).strip() for l in open(path))
    return [l for l in lines if l]


def block_after(lines, i):
    """The lines of the brace block that opens on line i."""
    depth, out = 0, []
    for l in lines[i:]:
        depth += l.count("{") - l.count("}")
        out.append(l)
        if depth <= 0:
            break
    return out


def refill_guards(lines):
    """Barriers that a single-thread role waits on before it starts copies into (or stores out of) shared memory."""
    names = set()
    for i, l in enumerate(lines):
        if "elect_one()" not in l or "{" not in l or l.startswith("__device__"):
            continue
        block = block_after(lines, i)
        if any("expect_tx(" in b or "tma_store_3d(" in b for b in block):
            names |= {m for b in block for m in re.findall(r"mbar_wait\(&(\w+)", b)}
    return names


@pytest.mark.parametrize("name,guards", [
    ("ssd_conv.cu", {"empty"}),
    ("ssd_tc_bcf.cu", {"rempty", "vempty", "stempty"}),
    ("ssd_tc_chain.cu", {"empty"}),
    ("ssd_tc_scan.cu", {"empty", "rowsfree", "xrempty", "outfull"}),
])
def test_readers_fence_before_they_give_a_buffer_back(name, guards):
    lines = statements(os.path.join(CSRC, name))
    assert refill_guards(lines) == guards
    for guard in guards:
        released = [i for i, l in enumerate(lines) if re.search(r"mbar_arrive\(&%s\b" % guard, l)]
        assert released or any("umma_commit(&%s" % guard in l for l in lines), guard
        for i in released:
            before = lines[max(0, i - 6):i]
            assert any(f in l for l in before for f in FENCED), (name, guard, before + [lines[i]])


def test_norm_rows_are_read_behind_a_fence_before_the_refill():
    # one CTA barrier per row gives the stage back; the thread behind it that starts the next copy has no fence of its own
    lines = statements(os.path.join(CSRC, "ssd_norm.cu"))
    refills = [i for i, l in enumerate(lines) if "issue(j + stages" in l]
    assert len(refills) == 1
    barrier = max(i for i in range(refills[0]) if lines[i].startswith("__syncthreads()"))
    assert lines[barrier - 1].startswith("fence_proxy_async_smem()")


def test_every_kernel_with_asynchronous_copies_is_looked_at():
    found = {os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu")) if any("expect_tx(" in l for l in statements(p))}
    assert found == {"ssd_conv.cu", "ssd_norm.cu", "ssd_tc_bcf.cu", "ssd_tc_chain.cu", "ssd_tc_scan.cu"}
