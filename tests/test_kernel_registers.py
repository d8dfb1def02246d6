"""Register bounds against the compiler's output (-Xptxas -v, kept by the build beside the objects): where
a pass states a bound, its kernels do not spill under it beyond what was measured to pay."""

import os
import re

import pytest

from paper_1712_00238_gb300 import build


def _spills():
    """{mangled kernel name: bytes of spill stores} of the library as built."""
    build.build()
    out = {}
    for f in sorted(os.listdir(build.OUT)):
        if not f.endswith(".ptxas"):
            continue
        with open(os.path.join(build.OUT, f)) as fh:
            text = fh.read()
        for m in re.finditer(r"Function properties for (\S+)\s+\d+ bytes stack frame, (\d+) bytes spill stores", text):
            out[m.group(1)] = int(m.group(2))
    return out


@pytest.fixture(scope="module")
def spills():
    s = _spills()
    assert len(s) > 300
    return s


def _named(spills, pattern):
    got = {k: v for k, v in spills.items() if re.search(pattern, k)}
    assert got, pattern
    return got


# FP32 column passes of the wide plan (32 columns a CTA), their half-spectrum form included
@pytest.mark.parametrize("pattern", [r"k_cols_halfIfLi(128|192|256|384)ELi\d+ELi32E", r"k_cols_fwd_pIfLi(128|192|256|384)ELi\d+ELi32E",
                                     r"k_cols_fused_pIfLi(128|192|256|384)ELi\d+ELi32E"])
def test_wide_plan_does_not_spill(spills, pattern):
    bad = {k: v for k, v in _named(spills, pattern).items() if v}
    assert not bad, bad


def test_row_pass_of_the_searches_does_not_spill(spills):
    # (precision, points, candidates kept) -> bytes that measured faster than a looser bound
    allowed = {("f", 192, 4): 400, ("d", 192, 1): 150, ("d", 192, 2): 150, ("d", 192, 4): 800}
    for name, n in _named(spills, r"k_rows_halfI[fd]Li\d+ELi\d+E").items():
        t, length, keep = re.search(r"k_rows_halfI([fd])Li(\d+)ELi(\d+)E", name).groups()
        assert n <= allowed.get((t, int(length), int(keep)), 64), (name, n)
