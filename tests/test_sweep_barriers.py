"""What the warps of a sweep block lower in shared memory has to be set before a barrier that
separates the two: a late store would undo a recorded minimum, and the unit's points would be
missing from a top-k list whose other entries are all right.  No run shows that reliably, so
the order is read from the source."""
import os
import re

SWEEP = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2601_02311_b200", "csrc", "ps_sweep.cu")


def kernel_source():
    text = open(SWEEP).read()
    text = re.sub(r"//[^\n]*", "", text)
    return text[text.index("k_sweep("):]


def test_lowest_cells_are_set_before_a_barrier():
    text = kernel_source()
    stores = [m.start() for m in re.finditer(r"sh\.least_cell\[[^\]]*\]\s*=[^=]", text)]
    first_item = text.index("atomicAdd(&sh.next1")         # the first pass begins
    assert stores and "atomicMin(&sh.least_cell[" in text
    for at in stores:
        assert "__syncthreads()" in text[at:first_item], "a store that the first pass's minima may race with"


def test_counters_of_the_passes_are_set_before_a_barrier():
    text = kernel_source()
    for name, use in (("next1", "atomicAdd(&sh.next1"), ("next2", "atomicAdd(&sh.next2"), ("full", "sh.full = 1")):
        at = re.search(rf"sh\.{name} = 0", text).start()
        assert "__syncthreads()" in text[at:text.index(use, at)], name
