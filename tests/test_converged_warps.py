"""Warp-wide tensor memory instructions (tcgen05.*.sync.aligned) are undefined unless all lanes execute them together.  Where code
in front of them branches by lane, that is left to the compiler unless the warp meets in between, so each stands behind a
__syncwarp() with no branch after it.  Checked on the sources: where lanes meet is the compiler's choice, and a wrong one need
not show."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2204_08400_b200", "csrc")
ALIGNED = re.compile(r'asm volatile\(\s*"tcgen05\.[^;]*?\.sync\.aligned')
BRANCH = re.compile(r"\b(if|else|while|do|switch|return|continue|break)\b|\?|&&|\|\|")  # loops with constant bounds are unrolled


def unsynchronised(text):
    """The start of every aligned tcgen05 statement with a branch between it and the last __syncwarp() (or without one)."""
    text = re.sub(r"//[^\n]*", "", text)
    bad = []
    for m in ALIGNED.finditer(text):
        met = text.rfind("__syncwarp();", 0, m.start())
        if met < 0 or BRANCH.search(re.sub(r'"[^"]*"', '""', text[met:m.start()])):
            bad.append(text[m.start():m.end()])
    return bad


@pytest.mark.parametrize("name", ["slonn_tile_kernels.cuh", "slonn_dense_tc.cu"])
def test_aligned_instructions_stand_behind_a_meeting_of_the_warp(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    assert ALIGNED.search(text)
    assert not unsynchronised(text)


def test_the_check_sees_what_is_missing():
    st = 'asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(a), "r"(b) : "memory");'
    assert unsynchronised("{ " + st + " }")
    assert unsynchronised("__syncwarp(); if (lane == 0) f(); " + st)
    assert not unsynchronised("__syncwarp(); " + st + "\n" + st)
    assert unsynchronised("__syncwarp(); " + st + " x = c ? 1 : 2; " + st)
