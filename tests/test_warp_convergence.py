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
        rest = re.sub(r"uint32_t r\[\d+\];|if constexpr \(!kTogether\) |__syncwarp\(\);", "", body)
        assert "__syncwarp();" in body and rest.strip() == "", stmt[:80]


# what only some lanes of a warp may do, or leave at different times
LANE_BRANCH = re.compile(r"\b(?:e|lane|tid|threadIdx\.x) (?:==|<)|\b(?:elect_one|warp_arrive|mbar_wait_bounded|\w+_wait|wait_cta)\b")


@pytest.mark.parametrize("name", [n for n in SOURCES if n.endswith(".cu")])
def test_loads_without_a_barrier_are_reached_together(name):
    """A load that leaves the barrier out (kTogether) follows a warp-wide
    barrier or vote, or a load that has one, with no branch of single lanes
    and no wait in between.  `load_sums` and `read_sums` (k_tensor_loop.cu)
    pass the demand on to their callers."""
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    text = re.sub(r"auto (?:load|read)_sums = .*?\n    \};\n", "", text, flags=re.S)
    for m in re.finditer(r"tmem_ld\w+<true>\(|\b(?:load|read)_sums\(", text):
        last = [k for k in re.finditer(r"__syncwarp\(\);|__all_sync\(.*?\);|tmem_ld\w+\(.*?\);", text[:m.start()], re.S)][-1]
        between = text[last.end():m.start()]
        assert not LANE_BRANCH.search(between), (name, between)


def test_the_wrappers_are_all_there():
    text = "".join(open(os.path.join(CSRC, n)).read() for n in SOURCES)
    assert len(list(_statements(text))) >= 15
