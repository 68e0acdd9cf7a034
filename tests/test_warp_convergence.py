"""Every inline-PTX statement with an `.aligned` instruction (all lanes of the
warp have to execute it together) is in a wrapper that brings the warp's lanes
together first (CPU: reads the sources)."""
import os
import re

import pytest

import paper_1905_00689_gb300 as package

CSRC = os.path.join(os.path.dirname(package.__file__), "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h")))


def _statements(text):
    """(statements before it in its function, statement) of each asm statement with `.aligned`."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"asm volatile\(", text):
        stmt = text[m.start():text.index(");\n", m.start())]
        if ".aligned" in stmt:
            yield text[text.rindex("__device__", 0, m.start()):m.start()], stmt


@pytest.mark.parametrize("name", SOURCES)
def test_aligned_instructions_follow_a_warp_barrier(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    found = list(_statements(text))
    assert sum(s.count(".aligned") for _, s in found) == re.sub(r"//[^\n]*", "", text).count(".aligned")
    for before, stmt in found:
        body = before[before.index("{") + 1:]
        # nothing but declarations and the barrier between the function's start and the instruction
        rest = re.sub(r"uint32_t r\[\d+\];|__syncwarp\(\);", "", body)
        assert "__syncwarp();" in body and rest.strip() == "", stmt[:80]


def test_the_wrappers_are_all_there():
    text = "".join(open(os.path.join(CSRC, n)).read() for n in SOURCES)
    assert len(list(_statements(text))) >= 15
