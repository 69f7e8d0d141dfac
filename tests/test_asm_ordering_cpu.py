"""Inline assembly that orders or performs memory accesses says so to the compiler.

An asm statement without a "memory" clobber may be passed by ordinary loads and stores: a read of words that an
asynchronous copy delivers could then be made before the wait for the copy.  Every statement of the CUDA sources
whose instructions copy asynchronously, wait, fence, signal a barrier, or touch tensor memory must carry the
clobber.  Checked on the source text: the fault it guards against is a race."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_13298_gb300", "csrc")
ORDERING = re.compile(r"cp\.async|mbarrier\.|fence\.|tcgen05\.(wait|commit|ld|st|mma|fence|alloc|dealloc|relinquish)")


def _statements(text):
    """(line, statement) of every asm statement, its parentheses matched outside string literals."""
    for m in re.finditer(r"\basm(?:\s+volatile)?\s*\(", text):
        depth, i, quoted = 1, m.end(), False
        while depth:
            c = text[i]
            if quoted and c == "\\":
                i += 1
            elif c == '"':
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            i += 1
        yield text.count("\n", 0, m.start()) + 1, text[m.start():i]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_ordering_asm_has_a_memory_clobber(path):
    with open(path) as f:
        # the run-time compiled kernel's source is text itself: its quotes are read as quotes
        text = f.read().replace('\\"', '"') if path.endswith("specialize.cu") else f.read()
    missing = [line for line, s in _statements(text) if ORDERING.search(s) and '"memory"' not in s]
    assert missing == []


def test_tensor_memory_loads_are_used_after_their_wait():
    """A tensor-memory load writes its registers up to the wait: the one place that waits names them as rewritten."""
    waits = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            text = f.read()
        n = text.count("tcgen05.wait::ld")
        if n:
            waits[os.path.basename(path)] = n
        if os.path.basename(path) != "tensor_core.cuh":
            assert not re.search(r"wait_ld\(\s*\)", text), path
    assert waits == {"tensor_core.cuh": 1}
    with open(os.path.join(CSRC, "tensor_core.cuh")) as f:
        body = f.read().split("void wait_ld(", 1)[1].split("\n}\n", 1)[0]
    assert '"+r"' in body
