"""Warp-private staging in shared memory (csrc/absorb.cu), read from the source: what the lanes of a
warp write in a lane-strided loop is read by other lanes, so a __syncwarp() stands between the loop
and the first read.  Reductions, ballots and shuffles order no memory between lanes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2310_10722_gb300", "csrc")
LOOP = re.compile(r"for \(int w = lane; [^;]*; w \+= 32\) \{")


def _block_end(text, at):
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced braces")


def _stagings():
    with open(os.path.join(CSRC, "absorb.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    for m in LOOP.finditer(text):
        end = _block_end(text, m.end() - 1)
        for name in re.findall(r"\b(\w+)\[w\] = ", text[m.end():end]):
            yield name, text[end:]


STAGINGS = list(_stagings())


def test_the_stagings_are_found():
    assert {n for n, _ in STAGINGS} >= {"lamv", "Tp", "Tm"}


@pytest.mark.parametrize("name,after", STAGINGS, ids=[f"{i}-{n}" for i, (n, _) in enumerate(STAGINGS)])
def test_staged_values_are_read_behind_a_warp_barrier(name, after):
    read = re.search(rf"\b{name}\b", after)
    assert read and "__syncwarp();" in after[:read.start()]
