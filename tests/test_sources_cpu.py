"""Properties of the CUDA sources that no run can show reliably."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_07814_gb300", "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            yield name, re.sub(r"//[^\n]*", "", f.read())


def test_tensor_memory_loads_reach_their_users_through_the_wait():
    """tcgen05.ld is asynchronous: its registers hold the values only after tcgen05.wait::ld.  A wait whose asm does not
    name them leaves the compiler free to place their first use before it, so each wait is followed by a
    statement that takes every loaded register as an operand."""
    waits = 0
    for name, text in _sources():
        for m in re.finditer(r"tcgen05\.wait::ld", text):
            waits += 1
            after = text[m.end():m.end() + 220]
            assert re.search(r'for \(int j = 0; j < (N|CH); \+\+j\) (\{\s*)?asm volatile\("" : "\+r"\(r\[j\]\)\);', after), (name, after)
    assert waits > 0
