"""Ring slots are handed back in order: a warp releases a slot of a shared-memory ring only
after a warp barrier, so that the copy that refills it cannot overtake a lane's last read.
Nothing on a GPU shows a missing barrier reliably, so the sources are read: every arrival
on an `empty` barrier goes through tc::ring_release, and that has the barrier first."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_00152_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def test_ring_slots_are_released_after_a_warp_barrier():
    released = 0
    for name, text in sources():
        assert not re.search(r"mbar_arrive\(\s*&?empty\s*\[", text), name
        released += len(re.findall(r"ring_release\(\s*&empty\[", text))
    assert released >= 3  # both ring kernels and the older TMA-fed one
    tc = dict(sources())["tc.cuh"]
    body = re.search(r"void ring_release\(uint64_t \*empty[^)]*\)\s*\{(.*?)\n\}", tc, re.S).group(1)
    assert re.search(r"^\s*__syncwarp\(\);.*mbar_arrive\(empty\)", body, re.S)
