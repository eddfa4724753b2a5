"""Rules of the kernels' hand-overs that no run can show broken, read off the sources (no GPU)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_18453_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def code(path):
    text = open(path).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_barrier_arrival_is_relaxed(path):
    # a relaxed arrival orders nothing that the arriving thread did before it
    assert "arrive.relaxed" not in code(path)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_aligned_barriers_follow_a_reconvergence(path):
    # bar.sync and barrier.cluster.arrive .aligned want whole warps, and the code before them branches by thread
    text = code(path)
    for m in re.finditer(r'asm volatile\(\s*"(bar\.sync|barrier\.cluster\.arrive)', text):
        assert re.search(r"__syncwarp\(\);\s*$", text[:m.start()]), text[m.start() - 80:m.end() + 40]


@pytest.mark.parametrize("path", [p for p in SOURCES if p.endswith(".cu")], ids=os.path.basename)
def test_kernels_with_bounded_waits_let_their_copies_land(path):
    # after an expired wait a kernel ends only when nothing is under way to its shared or tensor memory any more
    text = code(path)
    if re.search(r"tma_load_\w+\(|bulk_g2s\(|umma_\w+\(", text):
        assert "settle_after_timeout();" in text


@pytest.mark.parametrize("path", [p for p in SOURCES if p.endswith(".cu")], ids=os.path.basename)
def test_mmas_are_issued_by_the_elected_thread(path):
    # the block that an MMA stands in is entered by elect.sync, not by a comparison of the lane's number
    text = code(path)
    for m in re.finditer(r"\bumma_(f16|f16_c<\w+>|i8|commit)\(", text):
        entered = re.findall(r"if \((lane == 0|elect_one\(\))\) \{", text[:m.start()])
        assert entered and entered[-1] == "elect_one()", text[m.start() - 200:m.end()]
