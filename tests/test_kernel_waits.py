"""Waits inside kernels, by reading the sources: a wait that gives up after a limit leaves its kernel
with data that never came, so a kernel holding one has to report it.  The library's kernels report
through nothing but their outputs, and wait for copies by group counts and barriers, which end."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_00238_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_no_wait_that_gives_up(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    assert not re.search(r"\b(try_wait|test_wait)\b", text)
